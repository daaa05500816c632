"""The byte counts of the multigrid launches' profile: neighbour codes take two bytes a cell, group flags an
eighth of a byte, by the kernel that a level takes."""
import pytest

from paper_2603_21869_gb300 import binding, build, cases

pytestmark = pytest.mark.gpu


def per_cell(prof, site, cells):
    return prof[site]["bytes"] / prof[site]["launches"] / cells


def batch_profile(spec):
    build.ensure_built()
    with binding.Case(spec) as c, binding.Batch([c]) as b:
        b.step(1)
        return b.profile(1)


def test_batched_levels():
    """The batched kernels of whole quads: flags, and codes where the level has solid cells and the kernel
    does not go by the flags there (residual, restriction, inner products)."""
    spec = cases.heated_channel_3d(64, 32, 32, mg_levels=3, precision=cases.FP32, fixed_vcycles=2, krylov=1)
    box = [cases.Box(10, 16, 4, 10, 0, 7, thermal=cases.HEAT_FLUX, T_value=150.0)]
    N = 64 * 32 * 32
    for boxes, codes in (([], 0.125), (box, 2.0)):
        prof = batch_profile(spec.replace(boxes=boxes))
        assert per_cell(prof, "sweep_L0", N) == pytest.approx(3 * 4 + 0.125)
        assert per_cell(prof, "prolong_add_L0", N) == pytest.approx(2 * 4 + 4 / 8 + 0.125)
        assert per_cell(prof, "resid_restrict_L0", N) == pytest.approx(2 * 4 + 4 / 8 + codes)
        assert per_cell(prof, "resid0", N) == pytest.approx(8 + 4 + 2 * 4 + codes)
        assert 2 * per_cell(prof, "fcg_L0", N) == pytest.approx(6 * 4 + 16 + codes + 0.125)


def test_case_alone():
    """Under 2^20 cells alone: sweeps, transfers and the residual by the codes, the Krylov step by the flags."""
    build.ensure_built()
    spec = cases.heated_channel_3d(64, 32, 32, mg_levels=3, precision=cases.FP32, fixed_vcycles=2, krylov=1)
    N = 64 * 32 * 32
    with binding.Case(spec) as c:
        c.profile(True)
        c.step(1)
        prof = c.profile_read()
    assert per_cell(prof, "sweep_L0", N) == pytest.approx(3 * 4 + 2)
    assert per_cell(prof, "resid0", N) == pytest.approx(8 + 4 + 2 * 4 + 2)
    assert per_cell(prof, "fcg_L0", N) == pytest.approx(6 * 4 + 16 + 0.25)
