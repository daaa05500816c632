"""Clusters of 8, 4 and 2 blocks for the coarse levels (batches of nine, twenty and forty cases), and a plan
above the default shared-memory limit followed by a smaller one."""
import numpy as np
import pytest

from oracle.step import OracleCase
from paper_2603_21869_gb300 import binding, build, cases
from test_gpu_coarse import SHAPES

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.ensure_built()
    binding.lib()


@pytest.fixture(scope="module")
def stepped():
    """Cases with a flow, and the oracle's fields after one step of three V-cycles."""
    out = []
    for name in ("quads_aligned", "uneven_slabs", "rows_not_quads", "outlet_vents"):
        spec = SHAPES[name](precision=cases.FP64, fixed_vcycles=3, init_vel=(0.4, 0.3, 0.2), init_perturb=0.05, dt=1e-3)
        out.append((spec, OracleCase(spec).step(1).fields()))
    return out


@pytest.mark.parametrize("n", [9, 20, 40], ids=["8_blocks", "4_blocks", "2_blocks"])
def test_batched_steps_match_oracle(stepped, n):
    """FP64 within 1e-10 of the largest value, the bound of the parity tests (velocities: of the speed)."""
    cs = [binding.Case(stepped[i % len(stepped)][0]) for i in range(n)]
    try:
        binding.step_batch(cs, 1)
        got = [c.read() for c in cs]
    finally:
        for c in cs:
            c.close()
    for i, g in enumerate(got):
        want = stepped[i % len(stepped)][1]
        speed = max(float(np.max(np.abs(want[f]))) for f in ("u", "v", "w"))
        for f in cases.FIELDS:
            scale = speed if f in ("u", "v", "w") else float(np.max(np.abs(want[f])))
            assert float(np.max(np.abs(g[f] - want[f]))) <= 1e-10 * scale, (i, f)


def test_a_smaller_plan_does_not_lower_the_limit_of_a_larger_one():
    """The limit of dynamic shared memory belongs to the kernel: 65,536 FP32 cells of level 1 take about 65 KB
    a block of 16, the small case's levels less than the default 48 KB."""
    big_spec = cases.heated_channel_3d(128, 64, 64, mg_levels=5, precision=cases.FP32, fixed_vcycles=2, krylov=1)
    small_spec = cases.heated_channel_3d(32, 16, 16, mg_levels=3, precision=cases.FP32, fixed_vcycles=2, krylov=1)
    with binding.Case(big_spec) as big, binding.Case(small_spec) as small:
        small.step(1)
        assert big.step(2)["vcycles_last"] == 2
        with binding.Batch([small]) as b:
            b.step(1)
        with binding.Batch([big, small]) as b:
            b.step(1)
        big.step(1)
        assert np.isfinite(big.read(("p",))["p"]).all()
