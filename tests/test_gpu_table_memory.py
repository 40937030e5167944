"""The optional twiddle tables of double-precision transforms: sized by the passes
a plan can run, left out where they would take the memory other work needs, and
without influence on a plan's results."""
import numpy as np
import pytest

from paper_0901_1913_gb300 import synth

pytestmark = pytest.mark.gpu


def make(_fc2, N, **kw):
    c = synth.short_curve(seed=7, n=90)
    return _fc2.Plan(c.t, c.x, c.sigma, 2, 0.013, 9.0 / N, N, 2, "fp64", **kw)


@pytest.mark.parametrize("N,gridding", [(1 << 20, "kernel"), (1 << 22, "kernel"), (1 << 19, "paper")])
def test_tables_take_what_the_passes_need(N, gridding):
    from paper_0901_1913_gb300 import _fc2
    lib = _fc2.load()
    used = {}
    # the first plan also fills the library's cache of deconvolution tables
    for key, memory, tune in (("first", 1, True), ("none", 1, False), ("fixed", 0, False),
                              ("tuned", 0, True)):
        _fc2.table_memory(memory)
        try:
            before = lib.fc2_debug_pool_used(0)
            c = synth.short_curve(seed=7, n=90)
            f_min = 0.0 if gridding == "paper" else 0.013
            p = _fc2.Plan(c.t, c.x, c.sigma, 1, f_min, 9.0 / N, N, 2, "fp64", gridding=gridding,
                          autotune=tune)
            used[key] = lib.fc2_debug_pool_used(0) - before
            p.close()
        finally:
            _fc2.table_memory(0)
    M = 4 * N if gridding == "paper" else 2 * N
    # the last pass's table holds an entry per cell (16 bytes); a middle pass's is
    # that of its predecessors' radix product times its own, at most M / 2^7 here
    for key in ("fixed", "tuned"):
        extra = used[key] - used["none"]
        assert 16 * M <= extra <= 16 * (M + M // 64) + (1 << 16), (key, extra, M)


@pytest.mark.parametrize("N", [2048, 3001, 4096, 1 << 13, 1 << 14, 1 << 15, 50021, 1 << 17, 1 << 18,
                               1 << 19, 1 << 20, 1 << 22])
def test_plan_without_tables_gives_the_same_values(N):
    """Grids of 2^12 .. 2^23 points: every radix as a later pass, two and three passes."""
    from paper_0901_1913_gb300 import _fc2
    S = []
    for memory in (0, 1):
        _fc2.table_memory(memory)
        try:
            with make(_fc2, N) as p:
                d, _, _, _ = p.execute()
                S.append((p.spectra(), d))
        finally:
            _fc2.table_memory(0)
    np.testing.assert_array_equal(S[0][0], S[1][0])
    np.testing.assert_array_equal(S[0][1], S[1][1])


@pytest.mark.parametrize("N", [2048, 6001, 1 << 15, 1 << 18])
def test_batch_without_tables_matches_oracle(oracle_mod, N):
    from paper_0901_1913_gb300 import _fc2
    b = synth.survey_batch(seed=N % 97, C=3, N=N, T=50.0, f_max=1.0, n_median=60.0, n_hi=120)
    Hs = np.array([1, 2, 3], dtype=np.int32)
    df, f_min = 0.0013, 0.0604
    _fc2.table_memory(1)
    try:
        d, _, _ = _fc2.execute_batched(b.offsets, b.t, b.x, b.sigma, Hs, f_min, df, N, 2, "fp64",
                                       autotune="fixed")
    finally:
        _fc2.table_memory(0)
    bins = np.unique(np.concatenate([np.random.default_rng(N).integers(0, N, 120), [0, N - 1]]))
    at = 0
    for c in range(3):
        cur, H = b.curve(c), int(Hs[c])
        blk = d[at:at + H * N].reshape(H, N)
        at += H * N
        ref, piv = oracle_mod.dchi2_bins(cur.t, cur.x, cur.sigma, H, f_min, df, bins, with_pivots=True)
        _, _, chi0, _ = oracle_mod.moments(cur.x, cur.sigma)
        ok = piv >= 1e-4
        assert ok.sum() > 30
        # sums good to 1e-12 of W against such pivots, then a float result
        assert np.max(np.abs(blk[:, bins].T - ref)[ok]) <= 1e-6 * chi0
