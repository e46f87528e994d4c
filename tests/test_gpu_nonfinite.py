"""A NaN or an infinity in a digit-split product comes out as NaN where it has a
share in the result, and nowhere else."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


class OzSquare(ctypes.Structure):
    _fields_ = [("K", ctypes.c_int), ("Mp", ctypes.c_int), ("Krp", ctypes.c_int), ("e", ctypes.c_void_p),
                ("p", ctypes.c_void_p)]


@pytest.mark.parametrize("bad", [np.nan, 1j * np.inf, -np.inf])
@pytest.mark.parametrize("M,K", [(20, 70), (33, 300)])
def test_nonfinite_element_of_a_square_operand(M, K, bad):
    """Thin times Q and thin times Q^T on Q's digit planes split once (ozaki.cu):
    Q[3, 5] not finite makes column 5 of the one and column 3 of the other NaN;
    the other columns are the finite product to 1e-14 of its scale."""
    import torch
    from paper_1711_04798_gb300 import load_library
    lib = load_library()
    pack, thin = lib._Z14oz_pack_squareP11CUstream_stPK7double2iPvS4_P8OzSquareS6_, \
        lib._Z7oz_thinP11CUstream_stiPK7double2xbRK8OzSquarePS1_xbPvmPi
    size = lib._Z15oz_square_bytesi
    size.restype = ctypes.c_size_t
    ptr, i64 = ctypes.c_void_p, ctypes.c_longlong
    pack.argtypes = [ptr, ptr, ctypes.c_int, ptr, ptr, ptr, ptr]
    thin.argtypes = [ptr, ctypes.c_int, ptr, i64, ctypes.c_bool, ptr, ptr, i64, ctypes.c_bool, ptr, ctypes.c_size_t,
                     ptr]
    rng = np.random.default_rng(K)
    A = rng.standard_normal((M, K)) + 1j * rng.standard_normal((M, K))
    Q = rng.standard_normal((K, K)) + 1j * rng.standard_normal((K, K))
    Qb = Q.copy()
    Qb[3, 5] = bad
    dA, dQ = torch.tensor(A, device="cuda"), torch.tensor(Qb, device="cuda")
    mem = [torch.empty(size(K), dtype=torch.uint8, device="cuda") for _ in range(2)]
    work = torch.empty(64 << 20, dtype=torch.uint8, device="cuda")
    out = torch.zeros(M, K, dtype=torch.complex128, device="cuda")
    timeouts = torch.zeros(1, dtype=torch.int32, device="cuda")
    sq = [OzSquare(), OzSquare()]
    torch.cuda.synchronize()
    assert pack(None, dQ.data_ptr(), K, mem[0].data_ptr(), mem[1].data_ptr(), ctypes.addressof(sq[0]),
                ctypes.addressof(sq[1])) == 0
    for v, (ref, col) in enumerate(((Q, 5), (Q.T, 3))):
        assert thin(None, M, dA.data_ptr(), K, False, ctypes.addressof(sq[v]), out.data_ptr(), K, False,
                    work.data_ptr(), work.numel(), timeouts.data_ptr()) == 0
        torch.cuda.synchronize()
        C, scale = out.cpu().numpy(), np.abs(A) @ np.abs(ref)
        rest = np.arange(K) != col
        assert np.isnan(C[:, col]).all()
        assert (np.abs(C - A @ ref) / scale)[:, rest].max() < 1e-14
    assert timeouts.item() == 0
