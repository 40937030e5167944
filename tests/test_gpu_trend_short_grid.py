"""The gridded pass of the joint trend fit on both sides of the line between one
warp per trial frequency (short trial grids) and one thread, against the oracle."""
import numpy as np
import pytest

from paper_0901_1913_gb300 import synth
from tests.parity import compare

pytestmark = pytest.mark.gpu


# the line lies at 608 bins for three harmonics, 1216 for four to six, 1824 above
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("H,D,N", [(2, 3, 600), (3, 2, 608), (3, 3, 609), (4, 1, 1216), (4, 1, 1217),
                                   (5, 3, 1216), (5, 3, 1217), (6, 2, 31), (6, 2, 1400), (7, 2, 1824),
                                   (7, 2, 1825), (8, 1, 1824), (8, 1, 1825), (8, 3, 1800), (8, 3, 1900)])
def test_joint_solve_matches_oracle(oracle_mod, prec, H, D, N):
    from paper_0901_1913_gb300 import _fc2
    c = synth.short_curve(seed=H + 10 * D, n=350)
    u = c.t / 50.0 - 1.0
    x = c.x + 0.4 * u - 0.3 * u ** 2 + 0.2 * u ** 3
    f_min, df = 0.31, 0.0017
    d, _, _, chi0 = _fc2.periodogram(c.t, x, c.sigma, H, f_min, df, N, 2, prec, detrend=D,
                                     trend_fit=True)
    bins = np.unique(np.concatenate([np.random.default_rng(N).integers(0, N, 200), [0, N - 1]]))
    ref, chi0_or, piv = oracle_mod.dchi2_trend_bins(c.t, x, c.sigma, H, D, f_min, df, bins,
                                                    with_pivots=True)
    assert chi0 == pytest.approx(chi0_or, rel=1e-9)
    r = compare(d[:, bins].T, ref, piv, chi0_or)
    assert r["ok"], r
