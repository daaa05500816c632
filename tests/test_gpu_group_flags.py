"""The vector kernels by the flags of four-cell groups (and by the codes where cells are solid): rows
whose ends are outlets, outlets along y and z, boxes that cut groups or fill them, row lengths of
whole and half eight-cell groups.  Stepped as batches (the vector kernels at any size), with and
without solid cells in the batch, against the FP64 oracle: the reduced-precision bound of 1e-4 of
each field's largest value (velocities: of the largest speed); 1e-3 for p, which carries the FP32
rounding of the velocity (1e-7 of 2 m/s) through the cell size over dt (about 4 m/s): 1e-6 against
a largest p of 0.05."""
import numpy as np
import pytest

from oracle.step import OracleCase
from paper_2603_21869_gb300 import binding, build, cases

pytestmark = pytest.mark.gpu

OUT = cases.Patch(cases.OUTLET)


def channel(nx, ny, nz, flip=False, **kw):
    s = cases.heated_channel_3d(nx, ny, nz, mg_levels=3, init_perturb=0.02, fixed_vcycles=8, krylov=1, **kw)
    if flip:   # the inlet on x+, the outlet on x-
        faces = list(s.faces)
        faces[0], faces[1] = faces[1], faces[0]
        s = s.replace(faces=faces, init_vel=(-2.0, 0.0, 0.0))
    return s


PLAIN = [lambda **k: channel(40, 16, 12, **k), lambda **k: channel(36, 12, 16, flip=True, **k),
         lambda **k: channel(64, 8, 8, vents=[cases.Vent(3, 10, 23, 2, 6, OUT), cases.Vent(4, 33, 50, 0, 5, OUT)], **k)]
BOXED = [lambda **k: channel(40, 16, 12, boxes=[cases.Box(6, 17, 3, 9, 0, 5), cases.Box(24, 32, 8, 16, 4, 9)], **k),
         lambda **k: channel(48, 12, 16, flip=True, boxes=[cases.Box(13, 14, 2, 3, 0, 16)], **k)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.ensure_built()
    binding.lib()


@pytest.mark.parametrize("prec", [cases.FP32, cases.BF16_MIXED], ids=["fp32", "bf16"])
@pytest.mark.parametrize("group", [PLAIN, BOXED, PLAIN + BOXED], ids=["no_solids", "boxes", "mixed"])
def test_batched_steps_match_oracle(group, prec):
    specs = [make(precision=prec) for make in group]
    cs = [binding.Case(s) for s in specs]
    try:
        with binding.Batch(cs) as b:
            b.step(2)
        got = [c.read() for c in cs]
    finally:
        for c in cs:
            c.close()
    for i, (s, g) in enumerate(zip(specs, got)):
        ref = OracleCase(s).step(2).fields()
        speed = max(float(np.max(np.abs(ref[f]))) for f in ("u", "v", "w"))
        for f in cases.FIELDS:
            scale = speed if f in ("u", "v", "w") else float(np.max(np.abs(ref[f])))
            assert float(np.max(np.abs(g[f] - ref[f]))) <= (1e-3 if f == "p" else 1e-4) * scale, (i, f)
