"""The flexible-CG step of reduced-precision cases under 2^20 cells stepped alone forms its inner products,
its sums, alpha, beta and the step in FP64."""
import numpy as np
import pytest

from paper_2603_21869_gb300 import binding, build, cases

pytestmark = pytest.mark.gpu

PRECISIONS = pytest.mark.parametrize("prec", [cases.FP32, cases.BF16_MIXED], ids=["fp32", "bf16"])


def cube(prec, n=(64, 32, 32), **kw):
    """Cells of 1/8 (1/h^2 = 64 is exact in every type), walls and one outlet."""
    build.ensure_built()
    faces = [cases.Patch(cases.WALL)] * 6
    faces[1] = cases.Patch(cases.OUTLET)
    return cases.CaseSpec(nx=n[0], ny=n[1], nz=n[2], Lx=n[0] / 8, Ly=n[1] / 8, Lz=n[2] / 8, faces=faces, mg_levels=4,
                          precision=prec, krylov=1, init_k=1e-3, init_omega=1.0, **kw)


def solved(spec, b, cycles):
    with binding.Case(spec) as c:
        c.set_rhs(b)
        c.write({"p": np.zeros(b.shape)})
        c.vcycle(cycles)
        return c.read(("p",))["p"].copy()


@PRECISIONS
@pytest.mark.parametrize("smoother", [0, 1])
def test_scaled_right_hand_side_gives_scaled_pressure(prec, smoother):
    """A power of two on b is a power of two on p, to the bit: at 2^-70 every value is a normal FP32
    number, the products in the inner sums are not."""
    spec = cube(prec, smoother=smoother)
    b = np.random.default_rng(4).normal(size=(64, 32, 32)).astype(np.float32).astype(np.float64)
    p = solved(spec, b, 4)
    q = solved(spec, b * 2.0 ** -70, 4)
    assert np.any(p != 0.0)
    assert np.array_equal(q * 2.0 ** 70, p)


def apply_A(p):
    out = np.zeros_like(p)
    for a in range(3):
        g = np.pad(p, [(1, 1) if d == a else (0, 0) for d in range(3)], mode="edge")
        if a == 0:
            g[-1] = -g[-1]   # the outlet: p = 0 on the face
        lo, hi = np.take(g, range(0, p.shape[a]), axis=a), np.take(g, range(2, p.shape[a] + 2), axis=a)
        out += 64.0 * (2.0 * p - lo - hi)
    return out


def test_first_step_is_the_minimiser_along_its_direction():
    """After one iteration from zero p = alpha z with (b, z) = alpha (z, A z), so (b, p) = (p, A p): the
    relative difference is alpha's relative error.  The kernel forms A z in FP32: five operations a
    cell, 2^-24 of diag z each at random, ten standard deviations of their sum against (z, A z); b is rough, so
    that the sum is small against it.  An alpha in FP32 is off by up to 2^-24 beyond that: on nine
    right-hand sides and sweep counts it shows in seven."""
    for pre in (1, 2, 3):
        for post in (1, 2, 3):
            spec = cube(cases.FP32, fixed_vcycles=1, pre_sweeps=pre, post_sweeps=post)
            b = np.random.default_rng(3 * pre + post).normal(size=(64, 32, 32))
            b = (apply_A(apply_A(apply_A(b))) / 384.0 ** 3).astype(np.float32).astype(np.float64)
            p = solved(spec, b, 1)
            pAp = float(np.sum(p * apply_A(p)))
            tol = 10.0 * 5.0 * 2.0 ** -24 * 384.0 * float(np.sqrt(np.sum(p ** 4))) / pAp
            assert abs(float(np.sum(b * p)) - pAp) <= tol * pAp, (pre, post)
