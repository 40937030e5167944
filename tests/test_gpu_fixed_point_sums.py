"""The fixed-point sums of the last fix-up tier at every harmonic count (lanes
per multiple and tile lengths depend on it) and at sample counts around a tile
and a chunk, against the double tier."""
import numpy as np
import pytest

from paper_0901_1913_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H", [1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("n", [41, 255, 257, 4097, 5000])
def test_last_tier_matches_double_tier(H, n):
    from paper_0901_1913_gb300 import _fc2
    c = synth.short_curve(seed=n + H, n=n)
    bins = np.array([700, 1023, 4000, 9001, 16383])
    with _fc2.Plan(c.t, c.x, c.sigma, H, c.f_min, c.df, c.N, 2, "mixed") as p:
        _, _, _, chi0 = p.execute()
        d4 = p.exact_bins(bins, 4)
        d3 = p.exact_bins(bins, 3)
    # irregular times and n well above 2H + 1: relative pivots above 1e-4, so
    # sums good to 2^-45 give Delta chi^2 to 1e-9 chi2_0 with a wide margin
    assert np.max(np.abs(d4 - d3)) <= 1e-9 * chi0
