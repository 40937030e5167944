"""Sample sets whose fold wraps, at lengths around the run ordering's block and
its cap (longer sets, and those of many turns, take the radix sort), in both
precisions and in a batch of mixed lengths, against the oracle."""
import numpy as np
import pytest

from paper_0901_1913_gb300 import synth
from tests.parity import compare

pytestmark = pytest.mark.gpu


def check(oracle_mod, c, H, N, f_min, df, d):
    bins = np.unique(np.concatenate([np.random.default_rng(c.n).integers(0, N, 60), [0, N - 1]]))
    ref, piv = oracle_mod.dchi2_bins(c.t, c.x, c.sigma, H, f_min, df, bins, with_pivots=True)
    _, _, chi0, _ = oracle_mod.moments(c.x, c.sigma)
    r = compare(d[:, bins].T.astype(np.float64), ref, piv, chi0)
    assert r["ok"], r


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("n,turns", [(40, 40.0), (1023, 0.7), (1024, 1.6), (1025, 3.3), (2048, 9.2),
                                     (7167, 1.1), (7168, 2.4), (7169, 2.4),
                                     (700, 93.0), (3000, 400.0)])
def test_plan_matches_oracle(oracle_mod, prec, n, turns):
    from paper_0901_1913_gb300 import _fc2
    c = synth.short_curve(seed=n, n=n)
    H, N, df = 2, 700, turns / 100.0  # `turns` of the fold over the span at k = 1
    d, _, _, _ = _fc2.periodogram(c.t, c.x, c.sigma, H, 0.011, df, N, 2, prec)
    check(oracle_mod, c, H, N, 0.011, df, d)


def test_batch_matches_oracle(oracle_mod):
    from paper_0901_1913_gb300 import _fc2
    curves = [synth.short_curve(seed=i, n=n) for i, n in enumerate((30, 900, 1500, 7168, 7300, 41))]
    off = np.concatenate([[0], np.cumsum([c.n for c in curves])])
    t, x, s = (np.concatenate([getattr(c, k) for c in curves]) for k in ("t", "x", "sigma"))
    H, N, df = 2, 900, 0.013
    d, _, _ = _fc2.execute_batched(off, t, x, s, H, 0.02, df, N, 2, "mixed", autotune="fixed")
    for i, c in enumerate(curves):
        check(oracle_mod, c, H, N, 0.02, df, d[i * H * N:(i + 1) * H * N].reshape(H, N))
