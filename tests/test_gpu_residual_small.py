"""The allocation-free residual on grids of fewer items than warps and on grids with collapsed axes (taken as
the axes that are left), each face zero-value in turn: against the oracle, 1e-12 of the largest value."""
import ctypes as ct

import numpy as np
import pytest

from oracle.geometry import Level
from oracle.poisson import residual
from paper_2603_21869_gb300 import binding, build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(17, 17, 1), (31, 31, 31), (33, 1, 20), (1, 1, 50), (1, 40, 1), (1, 33, 9), (70, 1, 1),
                                   (1, 1, 1), (65, 40, 33)])
def test_residual_of_small_and_collapsed_grids(shape):
    torch = pytest.importorskip("torch")
    build.ensure_built()
    rng = np.random.default_rng(sum(shape))
    h = (0.05, 0.07, 0.11)
    p, b = rng.standard_normal(shape), rng.standard_normal(shape)
    dev = [torch.from_numpy(np.ascontiguousarray(a.transpose(2, 1, 0)).ravel()).cuda() for a in (p, b)]
    for face in range(6):
        mask = [int(f == face) for f in range(6)]
        faces = [np.full(tuple(n for a, n in enumerate(shape) if a != f // 2), bool(mask[f])) for f in range(6)]
        ref = residual(Level(shape, h, np.zeros(shape, dtype=bool), faces), p, b)
        r = torch.full_like(dev[0], float("nan"))
        norms = torch.full((2,), float("nan"), dtype=torch.float64, device="cuda")
        st = binding.lib().fvm_poisson_residual_static(
            ct.c_void_p(dev[0].data_ptr()), ct.c_void_p(dev[1].data_ptr()), *shape, (ct.c_double * 3)(*h),
            (ct.c_int32 * 6)(*mask), ct.c_void_p(r.data_ptr()), ct.c_void_p(norms.data_ptr()), None)
        assert st == binding.OK, binding.last_error()
        torch.cuda.synchronize()
        got = r.cpu().numpy().reshape(shape[2], shape[1], shape[0]).transpose(2, 1, 0)
        assert float(np.max(np.abs(got - ref))) <= 1e-12 * float(np.max(np.abs(ref))), face
        r2, b2 = norms.cpu().numpy()
        assert r2 == pytest.approx(float(np.sum(ref * ref)), rel=1e-12)
        assert b2 == pytest.approx(float(np.sum(b * b)), rel=1e-12)
