"""The precision form's Lanczos mat-vecs at sizes where the boundary tests do not
reach: several 2048-column chunks of x, whole groups of 128 columns and
remainders, with the operators' FP32 copies and, without room for them, without."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


class Result(ctypes.Structure):
    _fields_ = [(f, ctypes.c_int) for f in ("iters", "converged", "breakdown", "indefinite")]


def _hermitian(rng, n, values):
    """Q diag(values) Q^H on FP32 entries, Q a product of three reflections."""
    m = np.diag(values).astype(complex)
    for _ in range(3):
        v = rng.standard_normal(n) + 1j * rng.standard_normal(n)
        v /= np.linalg.norm(v)
        m -= 2.0 * np.outer(v, v.conj() @ m)
        m -= 2.0 * np.outer(m @ v, v.conj())
    m = 0.5 * (m + m.conj().T)
    return m.astype(np.complex64).astype(complex)


@pytest.mark.parametrize("n", [96, 129, 2048, 2177, 4225])
def test_leading_values_with_and_without_narrowed_copies(n):
    """A with 8 values above 0.3, spread to 1, over a tail below 0.01; B within 0.1 of
    the identity.  Both paths form the same FP32 products in the same order, so
    their Ritz values are the same bits; against LAPACK on A and B (FP32 entries)
    they keep 1e-5: 2^-23 of each narrowed x and product, over the 60 steps."""
    import torch
    from paper_1711_04798_gb300 import load_library
    lib = load_library()
    f, need = lib._Z15lanczos_leadingP11CUstream_stPK7double2S3_xiidmPS1_xPdbP13LanczosResult, \
        lib._Z18lanczos_work_elemsxi
    p, i64 = ctypes.c_void_p, ctypes.c_longlong
    need.argtypes, need.restype = [i64, ctypes.c_int], i64
    f.argtypes = [p, p, p, i64, ctypes.c_int, ctypes.c_int, ctypes.c_double, ctypes.c_uint64, p, i64, p,
                  ctypes.c_bool, p]
    rng = np.random.default_rng(n)
    k, steps = 8, 60
    A = _hermitian(rng, n, np.concatenate([np.linspace(1.0, 0.3, k), 0.01 * rng.uniform(0.0, 1.0, n - k)]))
    B = _hermitian(rng, n, 1.0 + 0.1 * rng.uniform(-1.0, 1.0, n))
    dA, dB = torch.tensor(A, device="cuda"), torch.tensor(B, device="cuda")
    base = need(n, steps)
    out = []
    for room in (base, base + n * n + 64):
        work = torch.zeros(room, dtype=torch.complex128, device="cuda")
        s = torch.zeros(k, dtype=torch.float64, device="cuda")
        res = Result()
        torch.cuda.synchronize()
        assert f(None, dA.data_ptr(), dB.data_ptr(), n, k, steps, 1e-7, 5, work.data_ptr(), room, s.data_ptr(), True,
                 ctypes.addressof(res)) == 0
        torch.cuda.synchronize()
        assert res.converged == k and not res.indefinite
        out.append((res.iters, s.cpu().numpy()))
        del work
    assert out[0][0] == out[1][0] and np.array_equal(out[0][1], out[1][1])
    L = torch.linalg.cholesky(dB)
    ref = torch.linalg.eigvalsh((L.mH @ dA @ L).cpu()).numpy()[::-1][:k]
    assert np.abs(out[0][1] / ref - 1).max() < 1e-5
