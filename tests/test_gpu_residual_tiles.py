"""fvm_poisson_residual_static at the edges of its tiles (31 cells a warp along x, four rows a thread,
4 to 32 planes an item): one item exactly, one cell more, rows and planes left over, collapsed axes,
zero-value faces on every side.  r and both norms against the oracle's r = b - A p, within 1e-12 of
the largest value (a dozen rounded FP64 operations a cell)."""
import ctypes as ct

import numpy as np
import pytest

from oracle.geometry import Level
from oracle.poisson import residual
from paper_2603_21869_gb300 import binding, build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(31, 4, 4), (32, 5, 33), (62, 8, 3), (63, 6, 41), (1, 9, 13), (95, 1, 7), (94, 35, 1),
                                   (160, 70, 50)])
@pytest.mark.parametrize("mask", [(0, 1, 1, 0, 0, 1), (1, 0, 0, 1, 1, 0)], ids=["hi_lo_hi", "lo_hi_lo"])
def test_residual_at_tile_edges(shape, mask):
    torch = pytest.importorskip("torch")
    build.ensure_built()
    rng = np.random.default_rng(sum(shape) + sum(mask))
    h = (0.05, 0.07, 0.11)
    faces = [np.full(tuple(n for a, n in enumerate(shape) if a != f // 2), bool(mask[f])) for f in range(6)]
    lev = Level(shape, h, np.zeros(shape, dtype=bool), faces)
    p, b = rng.standard_normal(shape), rng.standard_normal(shape)
    ref = residual(lev, p, b)
    dev = [torch.from_numpy(np.ascontiguousarray(a.transpose(2, 1, 0)).ravel()).cuda() for a in (p, b)]
    r = torch.full_like(dev[0], float("nan"))
    norms = torch.full((2,), float("nan"), dtype=torch.float64, device="cuda")
    st = binding.lib().fvm_poisson_residual_static(
        ct.c_void_p(dev[0].data_ptr()), ct.c_void_p(dev[1].data_ptr()), *shape, (ct.c_double * 3)(*h),
        (ct.c_int32 * 6)(*mask), ct.c_void_p(r.data_ptr()), ct.c_void_p(norms.data_ptr()), None)
    assert st == binding.OK, binding.last_error()
    torch.cuda.synchronize()
    got = r.cpu().numpy().reshape(shape[2], shape[1], shape[0]).transpose(2, 1, 0)
    assert float(np.max(np.abs(got - ref))) <= 1e-12 * float(np.max(np.abs(ref)))
    r2, b2 = norms.cpu().numpy()
    assert r2 == pytest.approx(float(np.sum(ref * ref)), rel=1e-12)
    assert b2 == pytest.approx(float(np.sum(b * b)), rel=1e-12)
