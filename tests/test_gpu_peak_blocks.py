"""Best bins and peaks of plans with few and with many search blocks (one CTA
per block and row, or per block), at bin counts around a block's edge, against
numpy on the plan's own periodogram."""
import numpy as np
import pytest

from paper_0901_1913_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,H", [(2, 1), (4095, 2), (4096, 3), (4097, 8), (40000, 4), (4864 * 2048, 1),
                                 (4096 * 2433, 1), (1 << 21, 8), (1 << 22, 8)])
def test_best_and_peaks_match_numpy(N, H):
    from paper_0901_1913_gb300 import _fc2
    c = synth.short_curve(seed=3, n=200)
    df = 9.0 / N
    with _fc2.Plan(c.t, c.x, c.sigma, H, 0.05, df, N, 2, "mixed", top_k=5) as p:
        d, best, peaks, _ = p.execute()
    for h in range(H):
        assert best[h]["j"] == int(np.argmax(d[h]))
    row = d[H - 1]
    up = np.concatenate([[True], row[1:] > row[:-1]])
    down = np.concatenate([row[:-1] >= row[1:], [True]])
    j = np.flatnonzero(up & down)
    want = j[np.lexsort((j, -row[j]))][:5]
    assert [r["j"] for r in peaks if r["j"] >= 0] == want.tolist()
