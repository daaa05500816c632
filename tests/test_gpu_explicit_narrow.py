"""The explicit stage where its tiles are not whole: rows of 32 cells and of 31 m + 1 (the last lane owns the
row's last cell), one row or two to a block (planes of constant y), and such cases in a batch, whose
blocks have eight rows of which some are not there.  Against the oracle on the same state, with the
bounds of the stage tests (test_gpu_explicit_tiles)."""
import numpy as np
import pytest

from oracle.step import OracleCase
from paper_2603_21869_gb300 import binding, build, cases
from test_gpu_coarse import box_case
from test_gpu_step_fourcell import STATE, gpu_state

pytestmark = pytest.mark.gpu

SHAPES = {"x32": ((32, 16, 8), 2), "x94": ((94, 8, 6), 2), "x126": ((126, 4, 4), 2),
          "y1": ((64, 1, 48), 4), "y1_x32": ((32, 1, 32), 3), "y2": ((32, 4, 16), 2), "x1": ((1, 32, 24), 3)}


def spec_of(name, prec, **kw):
    n, levels = SHAPES[name]
    axis = next(a for a in range(3) if n[a] > 1)
    vel = [0.0 if n[a] == 1 else 0.3 + 0.1 * a for a in range(3)]
    boxes = [cases.Box(0, max(1, n[0] // 8), 0, max(1, n[1] // 4), 0, max(1, n[2] // 4))]
    return box_case(n, levels, 2 * axis + 1, boxes, precision=prec, init_vel=tuple(vel), init_perturb=0.05, init_T=20.0,
                    fixed_vcycles=3, dt=1e-3, **kw)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.ensure_built()
    binding.lib()


@pytest.mark.parametrize("precision,tol", [(cases.FP32, 1e-5), (cases.FP64, 1e-12)], ids=["fp32", "fp64"])
@pytest.mark.parametrize("name", list(SHAPES))
def test_stage_of_incomplete_tiles(name, precision, tol):
    """Velocity components against the largest speed component (a plane's normal one is zero)."""
    spec = spec_of(name, precision)
    with binding.Case(spec) as c:
        c.step(1)
        c.run_stage(binding.STAGE_DT)
        dt = c.info()["dt"]
        x, p = gpu_state(c)
        c.run_stage(binding.STAGE_EXPLICIT)
        got = c.read(STATE)
    o = OracleCase(spec, state=x, p=p)
    o.dt = dt
    o.explicit()
    want = o.fields()
    speed = max(float(np.max(np.abs(want[f]))) for f in ("u", "v", "w"))
    for f in STATE:
        scale = speed if f in ("u", "v", "w") else float(np.max(np.abs(want[f])))
        assert float(np.max(np.abs(got[f] - want[f]))) <= tol * scale, f


def test_missing_rows_in_a_batch():
    """FP64: the batched stage does the same arithmetic (1e-12 after a step that depends on no solve)."""
    specs = [spec_of(name, cases.FP64) for name in SHAPES]
    alone = []
    for s in specs:
        with binding.Case(s) as c:
            c.step(1)
            alone.append(c.read(("T", "k", "omega")))
    cs = [binding.Case(s) for s in specs]
    try:
        binding.step_batch(cs, 1)
        got = [c.read(("T", "k", "omega")) for c in cs]
    finally:
        for c in cs:
            c.close()
    for name, g, a in zip(SHAPES, got, alone):
        for f in g:
            assert float(np.max(np.abs(g[f] - a[f]))) <= 1e-12 * float(np.max(np.abs(a[f]))), (name, f)
