"""Tile sizes and K splits of the FP64 CUDA-core GEMM, at the edges of its 16,
32 and 64 wide tiles, against numpy.  Sums of K products in any order stay
within (K + 2) eps of sum_k |A_ik| |B_kj|, with a factor sqrt(2) per complex
product."""
import numpy as np
import pytest

from test_gpu_tc_gemm import _op, _zgemm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 1), (16, 16, 8), (17, 33, 9), (24, 32, 32), (32, 64, 64), (48, 108, 108),
                                   (80, 1024, 1024), (65, 129, 31), (1000, 3, 17), (700, 650, 40)])
@pytest.mark.parametrize("ops", [(0, 0), (1, 3), (2, 1)])
def test_fp64_gemm_tiles(shape, ops):
    M, N, K = shape
    rng = np.random.default_rng(M + N + K)
    sa, sb = ((K, M) if ops[0] & 1 else (M, K)), ((N, K) if ops[1] & 1 else (K, N))
    A = rng.standard_normal(sa) + 1j * rng.standard_normal(sa)
    B = rng.standard_normal(sb) + 1j * rng.standard_normal(sb)
    C = _zgemm(0, A, ops[0], B, ops[1], M, N, K)
    a, b = _op(A, ops[0]), _op(B, ops[1])
    assert np.all(np.abs(C - a @ b) <= 2 * 1.42 * (K + 2) * 2.3e-16 * (np.abs(a) @ np.abs(b)))
