"""The 2^8, 2^9 and (first) 2^10 transform passes as first, middle and last passes, with grids
occupied in part (skipped zero levels) and throughout and trial grids of half
the modes and fewer: spectra against the radix-16 family's."""
import numpy as np
import pytest

from paper_0901_1913_gb300 import synth

pytestmark = pytest.mark.gpu


# grid lengths: 2^16 = 8 x 8, 2^17 = 9 x 8, 2^18 = 9 x 9, 2^25 = 9 x 8 x 8, 2^26 = 9 x 9 x 8
@pytest.mark.parametrize("N,oversample,fill", [
    (1 << 15, 2, 0.03), (1 << 15, 2, 0.3), (25001, 2, 0.11), (1 << 14, 4, 0.3),
    (1 << 16, 2, 0.005), (1 << 16, 2, 0.45), (50021, 2, 0.2), (1 << 15, 4, 0.24),
    (1 << 17, 2, 0.06), (1 << 17, 2, 0.49), (100003, 2, 0.13), (1 << 16, 4, 0.3),
    # 2^19 = 10 x 9 and 2^20 = 10 x 10: the 2^10 first pass, stored directly and staged
    (1 << 18, 2, 0.03), (1 << 18, 2, 0.1), (1 << 18, 2, 0.45), (200003, 2, 0.25), (1 << 17, 4, 0.2),
    (1 << 19, 2, 0.06), (400009, 2, 0.3), (1 << 24, 2, 0.2), (1 << 25, 2, 0.01)])
def test_spectra_match_radix16_family(N, oversample, fill):
    from paper_0901_1913_gb300 import _fc2
    c = synth.short_curve(seed=5, n=300)
    df = fill / 100.0  # occupied fraction of the first harmonic's grid
    f_min = df if oversample == 4 else 0.37 * df  # packed, and modulated grids
    S = {}
    for family in ("default", "r16"):
        with _fc2.Plan(c.t, c.x, c.sigma, 1, f_min, df, N, oversample, "mixed",
                       fft_kernel=family) as p:
            p.execute()
            S[family] = p.spectra()
    W = float(np.sum(c.sigma ** -2.0))
    d = np.abs(c.x - np.average(c.x, weights=c.sigma ** -2.0))
    scale = np.array([W, W, float(np.sum(d * c.sigma ** -2.0))])
    # each family's float transform is within 1e-6 of the terms' modulus sum
    # (a few roundings of each of log2 M levels); two of them within twice that
    err = np.max(np.abs(S["default"] - S["r16"]), axis=1) / scale
    assert np.all(err <= 2e-6), err
