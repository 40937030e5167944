"""The gridded pass of the joint trend fit at every harmonic count and degree
(its solve holds one trial frequency per thread; the counts decide its register
layout), with a trial grid one bin past a thread block."""
import numpy as np
import pytest

from paper_0901_1913_gb300 import synth
from tests.parity import compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("H,D", [(1, 1), (1, 3), (2, 2), (3, 1), (4, 2), (5, 3), (6, 1), (7, 2),
                                 (8, 1), (8, 3)])
def test_joint_solve_matches_oracle(oracle_mod, prec, H, D):
    from paper_0901_1913_gb300 import _fc2
    c = synth.short_curve(seed=H + 10 * D, n=350)
    u = c.t / 50.0 - 1.0
    x = c.x + 0.4 * u - 0.3 * u ** 2 + 0.2 * u ** 3
    N, f_min, df = 129, 0.31, 0.0113
    d, _, _, chi0 = _fc2.periodogram(c.t, x, c.sigma, H, f_min, df, N, 2, prec, detrend=D,
                                     trend_fit=True)
    bins = np.arange(N)
    ref, chi0_or, piv = oracle_mod.dchi2_trend_bins(c.t, x, c.sigma, H, D, f_min, df, bins,
                                                    with_pivots=True)
    assert chi0 == pytest.approx(chi0_or, rel=1e-9)
    r = compare(d.T, ref, piv, chi0_or)
    assert r["ok"], r
