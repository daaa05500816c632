"""The level-0 residual of reduced-precision cases under 2^20 cells stepped alone, at the floor that
V-cycles reach (r = b - A p of the size of p's last bits): its norm against the one formed in extended
precision from the same stored p and b.

Tolerance: with FP64 arithmetic a cell's r has three additions, three multiply-adds of the running
sum and a last one that cancels; at half a unit in the last place each (2^-53, taken as the standard
deviation) their root sum of squares s is the deviation of a cell's error.  A norm R of values with such
errors changes by |s|^2 / (2 R) and, at five standard deviations, by 5 |s| / sqrt(N).  r is then
rounded once to the corrections' storage (2^-24, 2^-9 for BF16, at random: over sqrt(N)), and
squared and summed in FP32 pairs (2^-22)."""
import numpy as np
import pytest

from paper_2603_21869_gb300 import binding, build, cases

pytestmark = pytest.mark.gpu


def walled_box(n, levels, **kw):
    faces = [cases.Patch(cases.WALL)] * 6
    faces[1] = cases.Patch(cases.OUTLET)
    return cases.CaseSpec(nx=n[0], ny=n[1], nz=n[2], Lx=0.1 * n[0], Ly=0.11 * n[1], Lz=0.12 * n[2], faces=faces,
                          mg_levels=levels, init_k=1e-3, init_omega=1.0, **kw)


def exact_residual(spec, p, b):
    """r = b - A p and the deviation of its FP64 evaluation, in extended precision."""
    P = p.astype(np.longdouble)
    r = b.astype(np.longdouble)
    ih = [np.float64(1.0) / (np.float64(L / n) ** 2) for L, n in ((spec.Lx, spec.nx), (spec.Ly, spec.ny), (spec.Lz, spec.nz))]
    for a in range(3):
        g = np.pad(P, [(1, 1) if d == a else (0, 0) for d in range(3)], mode="edge")
        if a == 0:
            g[-1] = -g[-1]   # the outlet: p = 0 on the face
        lo, hi = np.take(g, range(0, P.shape[a]), axis=a), np.take(g, range(2, P.shape[a] + 2), axis=a)
        r -= ((P - lo) + (P - hi)) * np.longdouble(ih[a])
    grow = np.cumsum(ih)
    s = 2.0 ** -53 * 2.0 * np.abs(p) * np.sqrt(sum(x * x for x in ih) + sum(x * x for x in grow))
    return r, s


@pytest.mark.parametrize("prec", [cases.FP32, cases.BF16_MIXED], ids=["fp32", "bf16"])
@pytest.mark.parametrize("n,levels", [((64, 32, 32), 4), ((36, 20, 24), 3)], ids=["rows_of_16", "ragged"])
def test_residual_norm_at_the_floor(prec, n, levels):
    build.ensure_built()
    spec = walled_box(n, levels, precision=prec)
    with binding.Case(spec) as c:
        c.set_rhs(np.random.default_rng(3).normal(size=n))
        c.vcycle(80)
        rel = c.vcycle(0)
        p, b = c.read(("p",))["p"], c.read_rhs()
    r, s = exact_residual(spec, p, b)
    norm = lambda x: float(np.sqrt(np.sum(x * x)))  # noqa: E731
    R, B, S, N = norm(r), norm(b), norm(s), r.size
    bits = 2.0 ** -24 if prec == cases.FP32 else 2.0 ** -9
    tol = S * S / (2.0 * R) + 5.0 * S / np.sqrt(N) + R * (bits * 5.0 / np.sqrt(N) + bits * bits + 2.0 ** -22)
    assert abs(rel * B - R) <= tol, (rel * B / R - 1.0, tol / R)
