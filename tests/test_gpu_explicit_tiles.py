"""The explicit stage at the edges of its tiles: warps of 31 cells, blocks of eight rows (two or four
on a 2D grid that would not fill the GPU), marches of several planes.

One stage is compared with the oracle's on the same state.  A cell's new value is its old one plus dt
times a sum of some forty products, each at most a Courant number (here below 1) times the field, so its
rounding is below 100 u of the field's largest magnitude, u = 2^-53 or 2^-24: 1e-12 in FP64, 1e-5 in
FP32 (as in the other stage tests).  In a batch the march is longer, since the other cases fill the GPU;
after one step T, k and omega do not depend on the pressure solve and agree with the case alone to
single rounding errors (1e-6)."""
import numpy as np
import pytest

from oracle.step import OracleCase
from paper_2603_21869_gb300 import binding, build, cases
from test_gpu_step_fourcell import STATE, box_channel, check, gpu_state, rel_err

pytestmark = pytest.mark.gpu

SIZES = [(62, 16, 8, 2), (64, 18, 6, 2), (28, 10, 10, 2), (64, 16, 512, 4)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.ensure_built()
    binding.lib()


def explicit_against_oracle(spec, tol, label):
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
    if tol == 1e-5:
        return check(got, want, STATE, label)
    for n in STATE:
        ref = want["u"] if n in ("u", "v", "w") else want[n]
        assert np.max(np.abs(got[n] - want[n])) <= tol * np.max(np.abs(ref)), (label, n)


@pytest.mark.parametrize("precision,tol", [(cases.FP32, 1e-5), (cases.FP64, 1e-12)])
@pytest.mark.parametrize("size", SIZES)
def test_stage_at_tile_edges(size, precision, tol):
    nx, ny, nz, lv = size
    explicit_against_oracle(box_channel(nx, ny, nz, lv, precision=precision), tol, f"{size}")


@pytest.mark.parametrize("shape", [(48, 20), (30, 8), (64, 34)])
def test_stage_with_few_rows_per_block(shape):
    spec = cases.channel_2d(shape[0], shape[1], 2, fixed_vcycles=3, init_perturb=0.05, precision=cases.FP64)
    explicit_against_oracle(spec, 1e-12, f"2d {shape}")


def test_march_with_a_remainder_in_a_batch():
    # 84 cases x 6 columns x 2 marches: eight planes, then the four that remain
    specs = [box_channel(64, 16, 12, 3).replace(seed=100 + q) for q in range(84)]
    cs = [binding.Case(s) for s in specs]
    try:
        with binding.Batch(cs) as b:
            b.step(1)
        for q in (0, 41, 83):
            got = cs[q].read(("T", "k", "omega"))
            with binding.Case(specs[q]) as a:
                a.step(1)
                want = a.read(("T", "k", "omega"))
            for n in got:
                assert rel_err(got[n], want[n]) <= 1e-6, (q, n)
    finally:
        for c in cs:
            c.close()
