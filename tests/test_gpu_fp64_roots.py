"""The FP64 reciprocals and roots of dfloat.h against exact rational arithmetic
and CUDA's own results, and the cluster Cholesky at the ends of the FP64 range."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = """
#include "dfloat.h"
__global__ void roots(const double* a, int n, double* o) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  o[i] = rcp64_normal(a[i]);
  o[n + i] = rsqrt64(a[i]);
  o[2 * n + i] = df_val(df_rsqrt(df_of(a[i])));
  o[3 * n + i] = 1.0 / a[i];
  o[4 * n + i] = rsqrt(a[i]);
}
extern "C" int run_roots(const double* a, int n, double* o) {
  roots<<<(n + 255) / 256, 256>>>(a, n, o);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    import torch
    from paper_1711_04798_gb300 import build
    d = tmp_path_factory.mktemp("roots")
    src, so = os.path.join(d, "roots.cu"), os.path.join(d, "roots.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", "-cudart", "static", "-o",
                    so, src], check=True)
    f = ctypes.CDLL(so).run_roots
    f.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p]

    def call(a):
        a = torch.tensor(np.asarray(a, dtype=np.float64), device="cuda")
        o = torch.zeros(5, a.numel(), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert f(a.data_ptr(), a.numel(), o.data_ptr()) == 0
        return o.cpu().numpy()
    return call


def _edges():
    near = [m * (1.0 + k * 2.0 ** -52) for m in (1.0, 1.5, 2.0, 3.0) for k in (-1, 0, 1)]
    return near + [2.0 ** e * m for e in (-1021, -1020, 1019, 1020) for m in (1.0, 1.25, 1.9999)]


def test_reciprocals_and_roots_within_their_bounds(run):
    """2^-52 of the value: half an ulp of the last FMA, a quarter at most from the
    rounding of a x in 1 - a x^2, the truncated series below 2^-60.  The double-float
    root: an FP32 correction of the seed below 2^-20 of it, rounded to 2^-24 thrice,
    and double-float products good to 2^-46: 2^-43 in all."""
    rng = np.random.default_rng(0)
    a = np.concatenate([rng.uniform(1.0, 4.0, 20000), np.exp2(rng.uniform(-1000.0, 1000.0, 5000)), _edges()])
    o = run(a)
    for x, r, q in zip(a, o[0], o[1]):
        f = Fraction(x)
        assert abs(Fraction(r) * f - 1) < Fraction(1, 2 ** 52)
        assert abs(Fraction(q) ** 2 * f - 1) < Fraction(1, 2 ** 51)
    b = np.concatenate([rng.uniform(1.0, 4.0, 20000), np.exp2(rng.uniform(-60.0, 60.0, 5000))])
    for x, q in zip(b, run(b)[2]):
        h = np.float32(x)
        f = Fraction(float(h)) + Fraction(float(np.float32(x - float(h))))
        assert abs(Fraction(q) ** 2 * f - 1) < Fraction(1, 2 ** 42)


def test_roots_outside_the_normal_range_and_negative_reciprocals(run):
    a = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, -1.0, 5e-324, 1e-310])
    o = run(a)
    np.testing.assert_array_equal(o[1], o[4])
    neg = run(-np.exp2(np.linspace(-900.0, 900.0, 777)))
    assert np.abs(neg[0] / neg[3] - 1).max() < 2.0 ** -51 and np.isnan(neg[1]).all()


@pytest.mark.parametrize("kind", ["graded", "small", "large"])
@pytest.mark.parametrize("n", [32, 57])
def test_cluster_cholesky_at_the_ends_of_the_range(n, kind):
    """R and R^{-H} of pivots that reach the subnormals (a diagonal matrix: roots
    alone, 4 eps) or lie at 2^-1018 and 2^1022 throughout (a dominant diagonal: n eps
    of the root's scale, computed on the scaled matrix by LAPACK)."""
    import torch
    from paper_1711_04798_gb300 import load_library
    f = load_library()._Z9chol_dropP11CUstream_stPK7double2PS1_S4_S4_id
    p = ctypes.c_void_p
    f.argtypes = [p, p, p, p, p, ctypes.c_int, ctypes.c_double]
    rng = np.random.default_rng(n)
    scale = {"graded": 0, "small": -1018, "large": 1022}[kind]
    if kind == "graded":
        base = np.diag(np.ldexp(rng.uniform(1.0, 2.0, n), np.linspace(-1060, 1020, n).astype(int))).astype(complex)
    else:
        base = 0.1 / n * (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))
        base = base + base.conj().T + 1.2 * np.eye(n)
    G = base if kind == "graded" else np.ldexp(base.real, scale) + 1j * np.ldexp(base.imag, scale)
    d = torch.tensor(G, device="cuda")
    w, R, L = (torch.zeros(n, n, dtype=torch.complex128, device="cuda") for _ in range(3))
    torch.cuda.synchronize()
    assert f(None, d.data_ptr(), w.data_ptr(), R.data_ptr(), L.data_ptr(), n, 0.0) == 0
    torch.cuda.synchronize()
    R, L = R.cpu().numpy(), L.cpu().numpy()
    eps = 2.3e-16
    if kind == "graded":
        r = np.sqrt(np.diag(G).real)
        assert np.abs(np.diag(R) / r - 1).max() < 4 * eps and np.abs(np.diag(L) * r - 1).max() < 4 * eps
        assert not np.any(R - np.diag(np.diag(R))) and not np.any(L - np.diag(np.diag(L)))
        return
    ref = np.linalg.cholesky(base).conj().T
    h = scale // 2
    assert np.abs(np.ldexp(R.real, -h) + 1j * np.ldexp(R.imag, -h) - ref).max() < n * eps
    assert np.abs(np.ldexp(L.real, h) + 1j * np.ldexp(L.imag, h) - np.linalg.inv(ref).conj().T).max() < n * eps
