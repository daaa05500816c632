"""fvm_lambda2 into pinned buffers that the kernel must not store into itself: they get the staging
copy's bytes, and nothing beside them changes."""
import numpy as np
import pytest

from paper_2603_21869_gb300 import binding, build, cases

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def case():
    build.ensure_built()
    with binding.Case(cases.heated_channel_3d(24, 16, 8, mg_levels=3, precision=cases.FP32, fixed_vcycles=2,
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
