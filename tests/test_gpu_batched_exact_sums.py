"""The exact sums of a batch's entries as one warp forms them, at every harmonic count
(lanes per multiple and staged tiles depend on it), in every capacity that holds
it, at sample counts around the tiles and the block pairs of the fixed-point tier,
against sums in extended precision."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def sums(A, B, wq, wp, j, H, capacity, tier):
    from paper_0901_1913_gb300 import _fc2
    fn = _fc2.load().fc2_debug_batch_sums
    p = ctypes.c_void_p
    fn.argtypes = [p, p, p, p, ctypes.c_int64, ctypes.c_int64, ctypes.c_int, ctypes.c_int,
                   ctypes.c_int, p]
    fn.restype = ctypes.c_int
    out = np.zeros(6 * capacity)
    rc = fn(A.ctypes.data, B.ctypes.data, wq.ctypes.data, wp.ctypes.data, A.size, j, H, capacity, tier,
            out.ctypes.data)
    assert rc == 0
    z = out[0::2] + 1j * out[1::2]
    return z[:2 * capacity], z[2 * capacity:]


def direct(u, w, k):
    a = (np.uint64(k) * u).astype(np.longdouble) * (np.longdouble(2.0) ** -63)  # half turns
    a *= np.longdouble("3.14159265358979323846264338327950288")
    w = w.astype(np.longdouble)
    return complex(np.sum(w * np.cos(a)), np.sum(w * np.sin(a)))


@pytest.mark.parametrize("H", [1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 64, 65, 127, 255, 257, 511, 513, 1025, 2047, 4099])
def test_one_warp_sums_match_extended_precision(H, n):
    rng = np.random.default_rng(100 * n + H)
    A, B = (rng.integers(0, 1 << 64, n, dtype=np.uint64) for _ in range(2))
    wq = np.exp(rng.normal(size=n)) * 400.0
    wp = wq * 0.3 * rng.normal(size=n)
    j = int(rng.integers(0, 1 << 24))
    u = A + np.uint64(j) * B
    Q = np.array([direct(u, wq, k) for k in range(1, 2 * H + 1)])
    P = np.array([direct(u, wp, k) for k in range(1, H + 1)])
    sq, sp = np.sum(wq), np.sum(np.abs(wp))
    # tier 4: phasors to 2^-46, products and block sums in double-float to 2^-46,
    # weights to 2^-48; the fixed point adds 2^-61 of the largest weight per block.
    # tier 3: up to 16 products of phasors and some 130 additions a lane in double
    for tier, tol in ((4, 2.0 ** -44), (3, 2.0 ** -45)):
        for capacity in (4, 6, 8):
            if capacity < H:
                continue
            q, p = sums(A, B, wq, wp, j, H, capacity, tier)
            assert np.max(np.abs(q[:2 * H] - Q)) <= tol * sq
            assert np.max(np.abs(p[:H] - P)) <= tol * sp
            assert not q[2 * H:].any() and not p[H:].any()
