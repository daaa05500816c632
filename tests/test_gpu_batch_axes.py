"""A batch of FP64 cases of which some have a collapsed x axis: their level-0 residual is another kernel, and
the loop goes on while any case of either kind iterates."""
import numpy as np
import pytest

from paper_2603_21869_gb300 import binding, build, cases

pytestmark = pytest.mark.gpu


def specs():
    faces = [cases.Patch(cases.EMPTY)] * 2 + [cases.Patch(cases.WALL)] * 4
    faces[3] = cases.Patch(cases.OUTLET)
    plane = cases.CaseSpec(nx=1, ny=64, nz=32, Lx=0.1, Ly=1.6, Lz=0.8, faces=faces, mg_levels=4, init_k=1e-3, init_omega=1.0,
                           init_vel=(0.0, 0.3, 0.0), init_perturb=0.05, mg_rel_tol=1e-9, max_vcycles=80, dt=1e-3)
    channel = cases.heated_channel_3d(32, 16, 16, mg_levels=3, init_perturb=0.02, mg_rel_tol=1e-4, max_vcycles=80)
    return [channel, plane, channel.replace(krylov=1, mg_rel_tol=1e-9)]


@pytest.mark.parametrize("order", [(0, 1, 2), (1, 0), (2, 1)], ids=str)
def test_batch_with_a_collapsed_x_axis(order):
    build.ensure_built()
    chosen = [specs()[i] for i in order]
    alone, counts = [], []
    for s in chosen:
        with binding.Case(s) as c:
            counts.append(c.step(3)["vcycles_total"])
            alone.append(c.read())
    cs = [binding.Case(s) for s in chosen]
    try:
        with binding.Batch(cs) as b:
            st = b.step(2)
            launches = b.info()["kernel_launches"]
            prof = b.profile(1)
            got = [c.read() for c in cs]
    finally:
        for c in cs:
            c.close()
    assert len(set(counts)) > 1 and launches > 0
    assert prof["resid0"]["launches"] % 2 == 0
    for i, (g, a) in enumerate(zip(got, alone)):
        speed = max(float(np.max(np.abs(a[f]))) for f in ("u", "v", "w"))
        for f in cases.FIELDS:
            scale = speed if f in ("u", "v", "w") else float(np.max(np.abs(a[f])))
            assert float(np.max(np.abs(g[f] - a[f]))) <= 1e-12 * scale, (i, f)
    assert len(st) == len(chosen)
