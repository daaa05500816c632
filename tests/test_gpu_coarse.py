"""The cluster kernel that cycles the coarse levels (csrc/coarse_kernels.cu) where its partition can
go wrong: levels dealt out in uneven slabs, coarse and fine slabs that do not line up, rows that are
not whole quads, two-dimensional levels in either plane, levels kept by one block, a hierarchy
whose only coarse level is the dense one, vents, boxes and a zero-value face on each axis.

Two V-cycles from zero on a random right-hand side against the oracle's: FP64 within 1e-10 of the
largest p (the FP64 bound of the parity tests: the same arithmetic in another order, about 1e2
rounded operations per value), FP32 corrections within 1e-4 (the reduced-precision bound)."""
import numpy as np
import pytest

from oracle.step import OracleCase
from paper_2603_21869_gb300 import binding, build, cases

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.ensure_built()
    binding.lib()


def box_case(n, levels, outlet, boxes=(), vents=(), **kw):
    """A walled box with one outlet face; axes of one cell are collapsed."""
    faces = [cases.Patch(cases.EMPTY if n[f // 2] == 1 else cases.WALL) for f in range(6)]
    faces[outlet] = cases.Patch(cases.OUTLET)
    return cases.CaseSpec(nx=n[0], ny=n[1], nz=n[2], Lx=0.1 * n[0], Ly=0.11 * n[1], Lz=0.12 * n[2], faces=faces,
                          mg_levels=levels, boxes=list(boxes), vents=list(vents), init_k=1e-3, init_omega=1.0, **kw)


B = cases.Box
OUT = cases.Patch(cases.OUTLET)
SHAPES = {
    "quads_aligned": lambda **k: box_case((64, 32, 32), 4, 1, [B(10, 23, 4, 17, 3, 11)], **k),
    "uneven_slabs": lambda **k: box_case((56, 40, 48), 4, 3, [B(0, 9, 30, 40, 20, 33)], **k),
    "slabs_out_of_step": lambda **k: box_case((48, 24, 72), 4, 4, [B(20, 28, 0, 9, 30, 50)], **k),
    "rows_not_quads": lambda **k: box_case((36, 20, 24), 3, 2, [B(5, 12, 6, 11, 0, 7)], **k),
    "more_planes_than_blocks": lambda **k: box_case((16, 16, 128), 3, 5, **k),
    "plane_xy": lambda **k: box_case((128, 64, 1), 4, 0, [B(30, 50, 8, 20, 0, 1)], **k),
    "plane_xz": lambda **k: box_case((64, 1, 96), 5, 5, **k),
    "plane_yz": lambda **k: box_case((1, 96, 32), 4, 3, **k),
    "line": lambda **k: box_case((512, 1, 1), 6, 1, **k),
    "dense_only": lambda **k: box_case((32, 16, 16), 2, 1, [B(6, 11, 2, 9, 0, 5)], **k),
    "one_block": lambda **k: box_case((24, 16, 8), 3, 1, **k),
    "outlet_vents": lambda **k: box_case((64, 48, 32), 4, 1, [B(30, 44, 10, 22, 0, 12)],
                                         [cases.Vent(4, 3, 9, 5, 11, OUT), cases.Vent(3, 40, 47, 20, 25, OUT)], **k),
}
SWEEPS = [(1, 1, 0), (2, 3, 1), (3, 2, 0)]   # pre, post, smoother


@pytest.mark.parametrize("prec,tol", [(cases.FP64, 1e-10), (cases.FP32, 1e-4)], ids=["fp64", "fp32"])
@pytest.mark.parametrize("name", list(SHAPES))
def test_vcycles_match_oracle(name, prec, tol):
    pre, post, smoother = SWEEPS[sorted(SHAPES).index(name) % 3]
    spec = SHAPES[name](precision=prec, pre_sweeps=pre, post_sweeps=post, smoother=smoother)
    o = OracleCase(spec)
    b = np.where(o.geo.fluid, np.random.default_rng(5).normal(size=o.geo.shape), 0.0)
    if prec == cases.FP32:
        b = b.astype(np.float32).astype(np.float64)
    p = np.zeros(o.geo.shape)
    for _ in range(2):
        p = o.mg.vcycle(p, b)
    with binding.Case(spec) as c:
        c.set_rhs(b)
        c.vcycle(2)
        got = c.read(("p",))["p"]
    assert float(np.max(np.abs(got - p))) <= tol * float(np.max(np.abs(p)))
