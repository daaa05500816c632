"""fvm_lambda2 into a pinned buffer (the kernel's own stores) and into a pageable one (a copy of the
staging buffer): the same bytes, boxes and collapsed axes included, nothing written past the field."""
import numpy as np
import pytest

from paper_2603_21869_gb300 import binding, build, cases

pytestmark = pytest.mark.gpu

BOX = cases.Box(5, 11, 3, 8, 0, 4, thermal=cases.HEAT_FLUX, T_value=80.0)


@pytest.mark.parametrize("prec", [cases.FP64, cases.FP32], ids=["fp64", "fp32"])
@pytest.mark.parametrize("shape", [(24, 16, 8), (36, 20, 1)], ids=["3d", "2d"])
def test_pinned_and_pageable_buffers_get_the_same_field(shape, prec):
    torch = pytest.importorskip("torch")
    build.ensure_built()
    if shape[2] == 1:
        spec = cases.channel_2d(shape[0], shape[1], 2, precision=prec, fixed_vcycles=2, init_perturb=0.05)
    else:
        spec = cases.heated_channel_3d(*shape, mg_levels=3, precision=prec, fixed_vcycles=2, init_perturb=0.05, boxes=[BOX])
    with binding.Case(spec) as c:
        c.step(2)
        pageable = np.full(c.N + 3, 7.0)
        c.lambda2(out=pageable[:c.N])
        pinned = torch.full((c.N + 3,), 7.0, dtype=torch.float64, pin_memory=True).numpy()
        c.lambda2(out=pinned[:c.N])
    assert np.array_equal(pinned, pageable)
    assert np.all(pinned[c.N:] == 7.0) and np.any(pinned[:c.N] != 0.0)
