"""V-cycles whose every level, the finest included, runs in one thread-block cluster and whose
correction is added to p there (small grids, one V-cycle per residual, no Krylov step): 3D rows of
whole quads and others, a plane of each orientation, uneven slabs, obstacles, vents, a zero-value face
on several axes, coarse sweeps equal to the fine ones, BF16 and FP32 corrections; and sizes just inside and
outside the cluster's limit.

Three V-cycles on a random right-hand side, with the p of one before the next, against the oracle's: FP64
within 1e-10 of the largest p, FP32 corrections within 1e-4 (the bounds of the coarse-level tests), BF16 corrections
within 2 % (eight bits in the stored residual, three times over).  Steps through the captured graph
give the fields of the stages run one by one."""
import numpy as np
import pytest

from oracle.step import OracleCase
from paper_2603_21869_gb300 import binding, build, cases
from test_gpu_coarse import B, OUT, box_case

pytestmark = pytest.mark.gpu

V = cases.Vent
SHAPES = {
    "quads": ((32, 16, 16), 3, dict(outlet=1, boxes=[B(6, 11, 2, 9, 0, 5)])),
    "uneven_slabs": ((24, 12, 20), 3, dict(outlet=4, boxes=[B(0, 5, 3, 8, 11, 17)])),
    "rows_not_quads": ((18, 14, 22), 2, dict(outlet=2, vents=[V(4, 3, 9, 5, 11, OUT)])),
    "plane_xy": ((128, 32, 1), 5, dict(outlet=0, boxes=[B(30, 50, 8, 20, 0, 1)])),
    "plane_xz": ((36, 1, 40), 3, dict(outlet=5)),
    "plane_yz": ((1, 64, 48), 4, dict(outlet=3)),
    "tiny": ((8, 4, 4), 2, dict(outlet=1)),
    "at_the_limit": ((32, 16, 16), 4, dict(outlet=3, pre_sweeps=2, post_sweeps=2, coarse_sweeps=2)),
    "past_the_limit": ((36, 16, 16), 3, dict(outlet=3)),
}
BOUND = {cases.FP64: 1e-10, cases.FP32: 1e-4, cases.BF16_MIXED: 2e-2}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.ensure_built()
    binding.lib()


def spec_of(name, prec, **kw):
    n, levels, d = SHAPES[name]
    d = dict(d)
    return box_case(n, levels, d.pop("outlet"), d.pop("boxes", ()), d.pop("vents", ()), precision=prec, krylov=0,
                    inner_cycles=1, **{**kw, **d})


@pytest.mark.parametrize("prec", list(BOUND), ids=["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("name", list(SHAPES))
def test_vcycles_match_oracle(name, prec):
    pre, post, smoother = [(1, 1, 0), (2, 3, 1), (3, 2, 0)][sorted(SHAPES).index(name) % 3]
    spec = spec_of(name, prec, pre_sweeps=pre, post_sweeps=post, smoother=smoother)
    o = OracleCase(spec)
    b = np.where(o.geo.fluid, np.random.default_rng(6).normal(size=o.geo.shape), 0.0)
    if prec != cases.FP64:
        b = b.astype(np.float32).astype(np.float64)
    p = np.zeros(o.geo.shape)
    for _ in range(3):
        p = o.mg.vcycle(p, b)
    with binding.Case(spec) as c:
        c.set_rhs(b)
        c.vcycle(3)
        got = c.read(("p",))["p"]
    assert float(np.max(np.abs(got - p))) <= BOUND[prec] * float(np.max(np.abs(p)))


def test_graph_steps_equal_stages():
    spec = cases.channel_2d(64, 32, 4, init_perturb=0.05, precision=cases.FP64)
    with binding.Case(spec) as a, binding.Case(spec) as b:
        a.step(3)
        for _ in range(3):
            for st in (binding.STAGE_DT, binding.STAGE_DESTRUCTION, binding.STAGE_EXPLICIT,
                       binding.STAGE_DESTRUCTION, binding.STAGE_RHS, binding.STAGE_SOLVE, binding.STAGE_PROJECT):
                b.run_stage(st)
        fa, fb = a.read(), b.read()
    for n in fa:
        scale = np.max(np.abs(fb["u"] if n in ("u", "v", "w") else fb[n]))
        assert np.max(np.abs(fa[n] - fb[n])) <= 1e-10 * scale, n
