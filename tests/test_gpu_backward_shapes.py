"""Gradients and refinement at every harmonic count, with sample counts at the
edges of the kernel's 128-thread passes and of the 2048 samples whose phasors
it keeps, against the oracle's gradients."""
import numpy as np
import pytest

from paper_0901_1913_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,n", [(1, 40), (2, 127), (3, 128), (4, 129), (5, 257), (6, 300),
                                 (7, 511), (8, 1000), (3, 2048), (2, 2200)])
def test_gradients_match_oracle(oracle_mod, H, n):
    from paper_0901_1913_gb300 import _fc2
    c = synth.short_curve(seed=H, n=n)
    f0 = c.truth["f0"]
    js = np.array([int(round((f - c.f_min) / c.df)) for f in (f0, 2 * f0, 3.1234)])
    g = np.array([1.0, -2.0, 0.5])
    with _fc2.Plan(c.t, c.x, c.sigma, H, c.f_min, c.df, c.N, 2, "mixed") as p:
        r = p.backward(js, grad_out=g)
    for k, j in enumerate(js):
        f = c.f_min + j * c.df
        _, gf, gx, gs = oracle_mod.grad(c.t, c.x, c.sigma, H, f)
        # double sums and an alpha of condition far below 1e7: rounding stays
        # below 1e-9 of the largest gradient
        assert r["d_df"][k] == pytest.approx(g[k] * gf, rel=1e-7, abs=1e-9 * abs(gf) + 1e-9)
        np.testing.assert_allclose(r["d_dx"][k], g[k] * gx, rtol=1e-7, atol=1e-9 * np.abs(gx).max())
        np.testing.assert_allclose(r["d_dsigma"][k], g[k] * gs, rtol=1e-7,
                                   atol=1e-9 * np.abs(gs).max())


def test_mixed_harmonic_counts_in_one_batch(oracle_mod):
    from paper_0901_1913_gb300 import _fc2
    b = synth.adjoint_batch(seed=9, C=8, n=150, N=1 << 12, T=50.0)
    H = np.arange(1, 9, dtype=np.int32)
    js = np.array([[int(round(t["f0"] / b.df[0])) - 1, 700] for t in b.truth])
    r = _fc2.backward_batched(b.offsets, b.t, b.x, b.sigma, H, b.f_min, b.df, b.N, js)
    for c in range(8):
        cur = b.curve(c)
        for k in range(2):
            f = cur.f_min + js[c, k] * cur.df
            _, gf, gx, gs = oracle_mod.grad(cur.t, cur.x, cur.sigma, int(H[c]), f)
            o = 2 * int(b.offsets[c]) + k * cur.n
            np.testing.assert_allclose(r["d_dx"][o:o + cur.n], gx, rtol=1e-7,
                                       atol=1e-9 * np.abs(gx).max())
            np.testing.assert_allclose(r["d_dsigma"][o:o + cur.n], gs, rtol=1e-7,
                                       atol=1e-9 * np.abs(gs).max())
