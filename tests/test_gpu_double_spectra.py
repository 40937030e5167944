"""Spectra of the double-precision transforms, in the plans' form and in the fused
form of the batches, against sums in extended precision: every radix of two- and
three-pass plans, grids occupied in part and throughout."""
import numpy as np
import pytest

from paper_0901_1913_gb300 import synth

pytestmark = pytest.mark.gpu

H = 2


def direct(c, t0, f):
    """Q_1..Q_2H and P_1..P_H at the frequencies f (extended precision)."""
    t = c.t.astype(np.longdouble) - np.longdouble(t0)
    w = c.sigma.astype(np.longdouble) ** -2
    xc = c.x - np.sum(w * c.x) / np.sum(w)
    turns = np.outer(f.astype(np.longdouble), t)
    rows = []
    for k, v in [(k, w) for k in range(1, 2 * H + 1)] + [(k, w * xc) for k in range(1, H + 1)]:
        a = 2 * np.pi * np.asarray(np.remainder(k * turns, 1), dtype=np.longdouble)
        rows.append(np.sum(v * np.cos(a), axis=1) + 1j * np.sum(v * np.sin(a), axis=1))
    scale = np.array([np.sum(w)] * (2 * H) + [np.sum(w * np.abs(xc))] * H, dtype=float)
    return np.array(rows), scale


# grids of 2^12 .. 2^24 points: 6 6, 7 6, 7 7, 8 7, 8 8, 9 8, 9 9, 10 9, 10 10, 11 10, 11 11,
# 8 8 7, 8 8 8
@pytest.mark.parametrize("N,fill", [(2048, 0.3), (3001, 0.02), (1 << 13, 0.45), (1 << 14, 0.1),
                                    (1 << 15, 0.4), (50021, 0.06), (1 << 17, 0.2), (1 << 18, 0.45),
                                    (1 << 18, 0.004), (1 << 19, 0.03), (1 << 20, 0.3),
                                    (1 << 20, 0.001), (1 << 21, 0.1), (4000001, 0.4),
                                    (4000001, 0.0003), (1 << 23, 0.0002)])
def test_spectra_match_extended_precision_sums(N, fill):
    from paper_0901_1913_gb300 import _fc2
    c = synth.short_curve(seed=N % 89, n=80)
    df = fill / 100.0
    f_min = 0.31 * df + 0.03
    bins = np.unique(np.concatenate([np.random.default_rng(N).integers(0, N, 60),
                                     [0, 1, N // 2 - 1, N // 2, N - 2, N - 1]]))
    with _fc2.Plan(c.t, c.x, c.sigma, H, f_min, df, N, 2, "fp64") as p:
        f = np.longdouble(f_min) + bins.astype(np.longdouble) * np.longdouble(df)
        ref, scale = direct(c, p.t0, f)
        p.execute()
        own = p.spectra()[:, bins]
        p.fused_passes(True)
        p.execute()
        fused = p.spectra()[:, bins]
        p.fused_passes(False)
        p.execute()
        again = p.spectra()[:, bins]
    # spreading and transform: 1e-12 of the weights.  A sample's phase k f tau carries
    # three roundings (tau, k df, their product), 2^-53 of the product each: up to
    # 4 2^-53 k f_max tau_max turns at the last modes, k = 2H, for every sample alike
    tol = 1e-12 + 2 * np.pi * 4 * 2.0 ** -53 * 2 * H * fill * N
    for S in (own, fused):
        assert np.max(np.abs(S - ref.astype(complex)) / scale[:, None]) <= tol
    np.testing.assert_array_equal(own, again)
