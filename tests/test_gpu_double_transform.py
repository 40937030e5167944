"""The fused double-precision transform passes of FP64 batches: every radix the
planner uses (grids of 2^12 .. 2^23 points), trial grids that keep exactly half
of the modes and fewer, and grids occupied in part (pruned first stages) and
throughout, against the oracle."""
import numpy as np
import pytest

from paper_0901_1913_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fill", [0.004, 0.06, 0.4])
@pytest.mark.parametrize("N", [2048, 4096, 6001, 16384, 30011, 65536, 131072, 262144, 524288,
                               1048576, 2000001, 4194304])
def test_fp64_batch_matches_oracle(oracle_mod, N, fill):
    from paper_0901_1913_gb300 import _fc2
    H, T = 2, 50.0
    b = synth.survey_batch(seed=N % 97, C=2, N=N, T=T, f_max=1.0, n_median=60.0, n_hi=120)
    df = fill / T                       # occupied fraction of the k = 1 grid
    f_min = 0.31 * df + 3.0 / T         # past the first few peaks of the window
    Hs = np.full(2, H, dtype=np.int32)
    d, _, _ = _fc2.execute_batched(b.offsets, b.t, b.x, b.sigma, Hs, f_min, df, N, 2, "fp64",
                                   autotune="fixed")
    bins = np.unique(np.concatenate([np.random.default_rng(N).integers(0, N, 120),
                                     [0, 1, N // 2 - 1, N // 2, N - 2, N - 1]]))
    for c in range(2):
        cur = b.curve(c)
        blk = d[c * H * N:(c + 1) * H * N].reshape(H, N)
        ref, piv = oracle_mod.dchi2_bins(cur.t, cur.x, cur.sigma, H, f_min, df, bins,
                                         with_pivots=True)
        _, _, chi0, _ = oracle_mod.moments(cur.x, cur.sigma)
        ok = piv >= 1e-6  # sums good to 1e-12 against pivots above 1e-6
        assert np.max(np.abs(blk[:, bins].T - ref)[ok], initial=0.0) <= 1e-5 * chi0
