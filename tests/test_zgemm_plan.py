"""Tile and K split of the FP64 CUDA-core GEMM, on the host."""
import ctypes

import pytest

UPPER = 1


def _plan(M, N, K, count=1, work=1 << 40, flags=0):
    from paper_1711_04798_gb300 import load_library
    f = load_library()._Z10zgemm_planiiiixiPiS_
    f.argtypes = [ctypes.c_int] * 4 + [ctypes.c_longlong, ctypes.c_int] + [ctypes.POINTER(ctypes.c_int)] * 2
    f.restype = None
    tile, ksplit = ctypes.c_int(), ctypes.c_int()
    f(M, N, K, count, work, flags, ctypes.byref(tile), ctypes.byref(ksplit))
    return tile.value, ksplit.value


@pytest.mark.parametrize("K", [1, 4, 7])
def test_short_sums_get_narrow_tiles_where_wide_ones_leave_sms_idle(K):
    """Below the splits' minimum of 8 too: 16 tiles of 64 for 1024 x 32, 128 of 16."""
    assert _plan(1024, 32, K) == (16, 0)
    assert _plan(16, 16, K) == (16, 0)
    assert _plan(64 * 152, 64 * 10, K) == (64, 0)  # waves of wide tiles: no narrow ones
    assert _plan(1024, 32, K, count=3) == (64, 0)  # batches keep theirs


def test_unsplit_hermitian_product_is_charged_its_full_square():
    """Without a split the tiles below the diagonal are computed as well, so
    without room for partials the choice is that of a general product."""
    for n in range(8, 400, 7):
        for K in (4, 15):  # unsplit
            assert _plan(n, n, K, flags=UPPER) == _plan(n, n, K)
