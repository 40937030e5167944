"""What launches each transform pass, as the host replay of the passes' indices
sees it: kernel, tile width, storing threads and store route.  The launcher asks
the same function, so the replay follows the kernels that run."""
import ctypes

import numpy as np
import pytest

SINGLE, R16, R64, BULK, R32, DUO, FIRST10, DOUBLE = range(8)
MODES, ROWS, STRIDE, BLOCKED, DIRECT = range(5)
DEFAULT, BULK_FAMILY, R16_FAMILY = 0, 3, 2


@pytest.fixture(scope="module")
def lib():
    import importlib
    importlib.import_module("paper_0901_1913_gb300.build").build()
    from paper_0901_1913_gb300 import _fc2
    L = _fc2.load()
    L.fc2_debug_fft_pass.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_void_p,
                                     ctypes.c_int, ctypes.c_int, ctypes.c_void_p]
    L.fc2_debug_fft_pass.restype = ctypes.c_int
    return L


def info(lib, rs, p, fp64=0, kernel=DEFAULT):
    r = np.ascontiguousarray(rs, dtype=np.int32)
    out = np.zeros(4, dtype=np.int32)
    rc = lib.fc2_debug_fft_pass(int(r.sum()), fp64, kernel, r.ctypes.data, r.size, p, out.ctypes.data)
    assert rc == 0, (rs, rc)
    return tuple(int(v) for v in out)


def test_first_pass_of_radix_2_10(lib):
    # three groups of 128 threads, each with a tile of 8 columns
    assert info(lib, [10, 9], 0) == (FIRST10, 3, 128, DIRECT)      # 2^19 points
    assert info(lib, [10, 10], 0) == (FIRST10, 3, 128, DIRECT)     # 2^20: the same layout
    assert info(lib, [10, 9, 9], 0) == (FIRST10, 3, 128, STRIDE)   # next tile: 16 columns
    # a next tile of 32 columns: 32 x 8 elements are more than a group's threads
    assert info(lib, [10, 8], 0) == (FIRST10, 3, 128, BLOCKED)
    # as a later pass, the register kernel on its 16-column tiles
    assert info(lib, [10, 10], 1) == (R64, 4, 256, MODES)
    assert info(lib, [10, 9], 0, kernel=BULK_FAMILY)[0] == BULK


def test_passes_of_radix_2_8_and_2_9(lib):
    assert info(lib, [9, 9], 0) == (DUO, 4, 256, ROWS)
    assert info(lib, [9, 9], 1) == (DUO, 4, 256, MODES)
    assert info(lib, [9, 9, 8], 0)[0] == DUO
    assert info(lib, [9, 9, 8], 1) == (DUO, 4, 256, DIRECT)        # a middle pass before the last
    assert info(lib, [9, 9], 0, kernel=R16_FAMILY)[0] == R16


def test_other_passes(lib):
    assert info(lib, [12, 12], 0) == (R64, 2, 256, ROWS)
    assert info(lib, [8, 7], 1) == (R16, 6, 512, MODES)
    assert info(lib, [11], 0)[::3] == (SINGLE, MODES)
    for rs in ([10, 9], [8, 8, 7]):
        for p in range(len(rs)):
            kind, logj, threads, route = info(lib, rs, p, fp64=1)
            assert (kind, logj, threads) == (DOUBLE, 12 - rs[p], 256)
            assert route == (MODES if p + 1 == len(rs) else ROWS if len(rs) == 2 else BLOCKED)
