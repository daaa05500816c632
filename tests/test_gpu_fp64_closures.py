"""The FP64 turbulence closures, which divide once a result, over the range of k and omega and past the
limits of their quotients (chi_k > 1e8, Re_t / R_beta > 1e4, chi_omega > 1e30, omega below its guard),
against the oracle, which divides as the formulas stand.

Each half step multiplies k and omega by a quotient whose limiters vary by less than their argument
does; an argument loses at most the cancellation of a sum of three products (here below 1e4) to
rounding: 1e-11 of the cell's own value.  In the explicit stage on a state uniform in k and omega the
production terms stand alone: 1e-12 of the field's largest value."""
import numpy as np
import pytest

from oracle.step import OracleCase, stable_dt, time_step
from paper_2603_21869_gb300 import binding, build, cases
from test_gpu_step_fourcell import STATE, gpu_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.ensure_built()
    binding.lib()


def channel(**kw):
    return cases.heated_channel_3d(32, 12, 8, mg_levels=2, precision=cases.FP64, init_perturb=0.05, **kw)


@pytest.mark.parametrize("k_exp,om_exp", [((-14, 3), (-8, 8)), ((-14, -10), (-13, -9)), ((0, 4), (-13, -6)),
                                          ((-2, 2), (-2, 2))])
def test_destruction_over_decades(k_exp, om_exp):
    spec = channel()
    rng = np.random.default_rng(7)
    shape = (spec.nx, spec.ny, spec.nz)
    with binding.Case(spec) as c:
        c.write({"u": 2.0 * rng.standard_normal(shape), "v": rng.standard_normal(shape),
                 "w": rng.standard_normal(shape), "k": 10.0 ** rng.uniform(*k_exp, shape),
                 "omega": 10.0 ** rng.uniform(*om_exp, shape)})
        c.run_stage(binding.STAGE_DT)
        dt = c.info()["dt"]
        x, p = gpu_state(c)
        c.run_stage(binding.STAGE_DESTRUCTION)
        got = c.read(("k", "omega"))
    o = OracleCase(spec, state=x, p=p)
    o.dt = dt
    o.destruction_half()
    want = o.fields()
    for n in got:
        assert np.max(np.abs(got[n] - want[n]) / np.abs(want[n])) <= 1e-11, n


@pytest.mark.parametrize("k0", [1e-14, 1e-6, 1.0, 1e3])
@pytest.mark.parametrize("om0", [1e-8, 1e-2, 1e4])
def test_production_and_time_step_bound(k0, om0):
    spec = channel(dt_adapt=True)
    rng = np.random.default_rng(8)
    shape = (spec.nx, spec.ny, spec.nz)
    with binding.Case(spec) as c:
        c.write({"u": 2.0 + rng.standard_normal(shape), "k": np.full(shape, k0), "omega": np.full(shape, om0)})
        c.run_stage(binding.STAGE_DT)
        dt = c.info()["dt"]
        x, p = gpu_state(c)
        c.run_stage(binding.STAGE_EXPLICIT)
        got = c.read(STATE)
    o = OracleCase(spec, state=x, p=p)
    assert abs(dt / stable_dt(o.geo, o.state, time_step(spec)) - 1.0) <= 1e-13
    o.dt = dt
    o.explicit()
    want = o.fields()
    for n in STATE:
        ref = want["u"] if n in ("u", "v", "w") else want[n]
        assert np.max(np.abs(got[n] - want[n])) <= 1e-12 * np.max(np.abs(ref)), n
