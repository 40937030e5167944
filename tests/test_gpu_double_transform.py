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


@pytest.mark.parametrize("N,fill", [(2048, 0.3), (6001, 0.02), (16384, 0.4), (30011, 0.1), (65536, 0.05),
                                    (131072, 0.2), (262144, 0.45), (524288, 0.03), (1048576, 0.1),
                                    (2000001, 0.3), (8388608, 0.02)])
def test_fp64_plan_matches_oracle(oracle_mod, N, fill):
    """Plans keep the passes' operation order, with tabled inter-pass twiddles
    and skipped zeros (2^12 .. 2^24 points, two and three passes)."""
    from paper_0901_1913_gb300 import _fc2
    c = synth.short_curve(seed=N % 89, n=80)
    H, df = 2, fill / 100.0
    f_min = 0.31 * df + 0.03
    d, _, _, chi0 = _fc2.periodogram(c.t, c.x, c.sigma, H, f_min, df, N, 2, "fp64")
    bins = np.unique(np.concatenate([np.random.default_rng(N).integers(0, N, 150),
                                     [0, 1, N // 2 - 1, N // 2, N - 2, N - 1]]))
    ref, piv = oracle_mod.dchi2_bins(c.t, c.x, c.sigma, H, f_min, df, bins, with_pivots=True)
    ok = piv >= 1e-4  # sums good to 1e-11 of W (phases up to 1e5 turns) against such pivots
    assert np.max(np.abs(d[:, bins].T - ref)[ok], initial=0.0) <= 1e-6 * chi0
