"""Which bins of a double-precision call are recomputed from exact sums: those whose
error estimate, from the largest coefficient norm of the nested models, is beyond
the bar.  The solves form the norm in float; here it is formed in double from direct
sums, with the rule's constants, over trial grids that run into singular equations
(frequencies below one turn over the span)."""
import numpy as np
import pytest

from paper_0901_1913_gb300 import synth

pytestmark = pytest.mark.gpu

TAU, EPS, BAR = 1e-9, 1e-13, 2e-5  # smallest relative pivot kept, error of a sum, the bar


def estimate(t, x, sigma, t0, H, f_min, df, N, tau):
    """The error estimate per bin when pivots above tau are kept (which columns those
    are depends on the phases' origin t0)."""
    w = sigma ** -2.0
    W = w.sum()
    xc = x - (w * x).sum() / W
    chi0 = (w * xc * xc).sum()
    z1 = np.exp(2j * np.pi * np.outer(f_min + df * np.arange(N), t - t0))
    q = np.ones((2 * H + 1, N), complex)
    p = np.zeros((H + 1, N), complex)
    z = np.ones_like(z1)
    for k in range(1, 2 * H + 1):
        z = z * z1
        q[k] = z @ w / W
        if k <= H:
            p[k] = z @ (w * xc) / np.sqrt(W * chi0)
    m = 2 * H + 1

    def alpha(l, k):
        hl, hk = (l + 1) // 2, (k + 1) // 2
        if k == 0:
            return q[hl].imag if l & 1 else q[hl].real
        d, s, sign = q[abs(hl - hk)], q[hl + hk], np.sign(hl - hk)
        if l & 1 and k & 1:
            return 0.5 * (d.real - s.real)
        if not l & 1 and not k & 1:
            return 0.5 * (d.real + s.real)
        return 0.5 * (s.imag + (sign if l & 1 else -sign) * d.imag)

    L = np.zeros((N, m, m))
    inv, zz = np.zeros((N, m)), np.zeros((N, m))
    for l in range(m):
        for k in range(l):
            L[:, l, k] = (alpha(l, k) - np.einsum("np,np->n", L[:, l, :k], L[:, k, :k])) * inv[:, k]
        a = alpha(l, l)
        d = a - np.einsum("np,np->n", L[:, l, :l], L[:, l, :l])
        keep = (a > 0) & (d > tau * a)
        inv[:, l] = np.where(keep, 1 / np.sqrt(np.where(keep, d, 1.0)), 0.0)
        h = (l + 1) // 2
        b = np.zeros(N) if l == 0 else (p[h].imag if l & 1 else p[h].real)
        zz[:, l] = (b - np.einsum("np,np->n", L[:, l, :l], zz[:, :l])) * inv[:, l]
    norm = np.zeros(N)
    for mp in range(3, m + 1, 2):
        A = np.zeros((N, mp))
        for l in range(mp - 1, -1, -1):
            A[:, l] = (zz[:, l] - np.einsum("np,np->n", L[:, l + 1:mp, l], A[:, l + 1:])) * inv[:, l]
        norm = np.maximum(norm, np.einsum("np,np->n", A, A))
    return EPS * (m * norm + 2 * np.sqrt(m * norm))


def bounds(*args):
    """Bins surely beyond the bar, and bins that may be.  The float back-substitution
    of a bin at the bar: at most some 17 2^-22 of the norm times the condition of L,
    itself about |A| there (5e3): 2%; the sums' own errors change it by 1e-4, and
    may keep or drop a column whose pivot is near the smallest one kept."""
    est = np.stack([estimate(*args, tau) for tau in (0.5 * TAU, TAU, 2.0 * TAU)])
    return int(np.all(est > 1.03 * BAR, axis=0).sum()), int(np.any(est > 0.97 * BAR, axis=0).sum())


@pytest.mark.parametrize("H", [2, 3, 4, 6, 8])
def test_plan_recomputes_the_bins_beyond_the_bar(H):
    from paper_0901_1913_gb300 import _fc2
    c = synth.short_curve(seed=H, n=300)
    N, df = 4096, 2.0 / (c.t.max() - c.t.min()) / 4096
    with _fc2.Plan(c.t, c.x, c.sigma, H, 3.3 * df, df, N, 2, "fp64") as p:
        p.execute()
        flagged, t0 = p.flag_count, p.t0
    lo, hi = bounds(c.t, c.x, c.sigma, t0, H, 3.3 * df, df, N)
    assert 20 < lo <= hi < 2 * lo  # the grid does run into the bar
    assert lo <= flagged <= hi
