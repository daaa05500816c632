"""A batched case's results, to the bit, whatever it shares the batch with: one other case or many (the
cluster of its coarse levels has 16, 8, 4 or 2 blocks, the columns of its level-0 reductions could follow
the number of cases) and cases with or without solid cells (the kernels by group flags and by codes)."""
import numpy as np
import pytest

from paper_2603_21869_gb300 import binding, build, cases

pytestmark = pytest.mark.gpu

BOX = [cases.Box(10, 16, 4, 10, 0, 7, thermal=cases.HEAT_FLUX, T_value=150.0)]


def small(i, prec, boxes):
    return cases.heated_channel_3d(32, 16, 16, mg_levels=3, precision=prec, seed=50 + i, init_perturb=0.02,
                                   mg_rel_tol=1e-6, max_vcycles=40, boxes=BOX if boxes else [])


PROBES = {   # level 1 between what a cluster of 8 and one of 16 blocks take alone
    "channel_fp32": lambda: cases.heated_channel_3d(128, 64, 64, mg_levels=5, precision=cases.FP32, init_perturb=0.02,
                                                    krylov=1, smoother=1, mg_rel_tol=1e-6, max_vcycles=60),
    "room_bf16": lambda: cases.room_3d(112, 80, 48, seed=3, mg_levels=4, h=0.04, precision=cases.BF16_MIXED, krylov=1,
                                       pre_sweeps=2, post_sweeps=2, inner_cycles=2, mg_rel_tol=1e-6, max_vcycles=60),
    # (in clusters of four blocks the right-hand side and the codes of level 1 stay in global memory)
    "channel_bf16": lambda: cases.heated_channel_3d(128, 64, 64, mg_levels=5, precision=cases.BF16_MIXED, init_perturb=0.02,
                                                    inner_cycles=2, mg_rel_tol=1e-6, max_vcycles=60),
    "channel_fp64": lambda: cases.heated_channel_3d(64, 32, 32, mg_levels=4, precision=cases.FP64, init_perturb=0.02,
                                                    mg_rel_tol=1e-6, max_vcycles=60),
}
COMPANIES = [(1, False), (1, True), (7, False), (7, True), (19, True), (40, False)]   # others, the first with a box


@pytest.mark.parametrize("name", list(PROBES))
def test_same_bits_in_every_batch(name):
    build.ensure_built()
    probe = PROBES[name]()
    seen = []
    for others, boxes in COMPANIES:
        specs = [small(i, probe.precision, boxes and i == 0) for i in range(others)] + [probe]
        cs = [binding.Case(s) for s in specs]
        try:
            with binding.Batch(cs) as b:
                st = b.step(3)[-1]
            seen.append((st["vcycles_total"], cs[-1].read()))
        finally:
            for c in cs:
                c.close()
    for (n, f), company in zip(seen[1:], COMPANIES[1:]):
        assert n == seen[0][0], company
        for x in cases.FIELDS:
            assert np.array_equal(f[x], seen[0][1][x]), (company, x)


@pytest.mark.parametrize("others", [0, 8], ids=["one", "nine"])
def test_bf16_batch_equals_the_case_alone(others):
    """The bounds that FP32 cases have against themselves alone (every solve to 1e-8): 1e-4 of the largest p, 1e-5
    of the other fields."""
    build.ensure_built()
    spec = cases.room_3d(64, 64, 32, seed=3, mg_levels=4, h=0.08, precision=cases.BF16_MIXED, krylov=1, pre_sweeps=2,
                         post_sweeps=2, inner_cycles=2, mg_rel_tol=1e-8, max_vcycles=80)
    with binding.Case(spec) as c:
        c.step(4)
        alone = c.read()
    cs = [binding.Case(s) for s in [small(i, spec.precision, i == 0) for i in range(others)] + [spec]]
    try:
        with binding.Batch(cs) as b:
            b.step(4)
        got = cs[-1].read()
    finally:
        for c in cs:
            c.close()
    speed = max(float(np.max(np.abs(alone[f]))) for f in ("u", "v", "w"))
    for f in cases.FIELDS:
        scale = speed if f in ("u", "v", "w") else float(np.max(np.abs(alone[f])))
        assert float(np.max(np.abs(got[f] - alone[f]))) <= (1e-4 if f == "p" else 1e-5) * scale, f
