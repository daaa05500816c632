"""fvm_lambda2 into pinned buffers that the kernel must not store into itself: they get the staging
copy's bytes, and nothing beside them changes."""
import numpy as np
import pytest

from paper_2603_21869_gb300 import binding, build, cases

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def case():
    build.ensure_built()
    with binding.Case(cases.heated_channel_3d(48, 32, 16, mg_levels=3, precision=cases.FP32, fixed_vcycles=2,
                                              init_perturb=0.05)) as c:
        c.step(2)
        yield c, c.lambda2().transpose(2, 1, 0).reshape(-1).copy()


@pytest.mark.parametrize("offset", [1, 4])
def test_unaligned_pinned_buffer(case, offset):
    torch = pytest.importorskip("torch")
    c, want = case
    raw = torch.full((8 * c.N + 16,), 7, dtype=torch.uint8, pin_memory=True).numpy()
    out = raw[offset:offset + 8 * c.N].view(np.float64)
    c.lambda2(out=out)
    assert np.array_equal(out, want)
    assert np.all(raw[:offset] == 7) and np.all(raw[offset + 8 * c.N:] == 7)


def test_buffer_between_two_registrations(case):
    """Both ends pinned, pageable memory between them: the kernel stores into neither.  The copy may
    refuse such a buffer, and the case stays usable."""
    torch = pytest.importorskip("torch")
    c, want = case
    page, N = 65536, 8 * c.N
    raw = np.full(N + 4 * page, 7, dtype=np.uint8)
    base = -(-raw.ctypes.data // page) * page
    at = base + page - 64                                        # the first 64 bytes in one registration ..
    far = (at + N - 1) // page * page
    assert base + page < far                                     # .. the last bytes in another, a gap between
    rt = torch.cuda.cudart()
    assert int(rt.cudaHostRegister(base, page, 0)) == 0 and int(rt.cudaHostRegister(far, page, 0)) == 0
    out = raw[at - raw.ctypes.data:][:N].view(np.float64)
    try:
        c.lambda2(out=out)
        assert np.array_equal(out, want)
    except binding.FvmError as e:
        assert e.status == binding.ERR_CUDA
    finally:
        assert int(rt.cudaHostUnregister(base)) == 0 and int(rt.cudaHostUnregister(far)) == 0
    assert np.array_equal(c.lambda2().transpose(2, 1, 0).reshape(-1), want)
