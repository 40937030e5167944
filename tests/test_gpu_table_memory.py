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
