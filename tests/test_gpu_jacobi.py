"""The cluster Jacobi SVD at the edges of its register tiles, schedules and
cluster sizes, through the entry points that run it."""
import numpy as np
import pytest

import oracle as O
import synth
from gpu_common import gpu_ctm

pytestmark = pytest.mark.gpu

EPS = 2.220446049250313e-16


def _corner(rng, n, kind):
    """A corner matrix: dense, graded over eight decades, or with rows of zeros
    and of rounding noise (rows that the schedule leaves out)."""
    m = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    if kind == "graded":
        d = np.logspace(0, -8, n)
        m = d[:, None] * m * d[None, :]
    if kind == "sparse":
        m[n // 3 : n // 2] = 0.0
        m[n // 2 : n // 2 + 2] *= 1e-17
    return m


@pytest.mark.parametrize("n", [8, 31, 32, 33, 65, 127, 128, 129, 250, 256, 257, 300])
def test_corner_spectra_against_lapack(n):
    """Sixteen corners at once (one launch, a cluster each, from n = 32; one
    after another below), against LAPACK.  A Jacobi that stops at inner products of n eps
    leaves errors of order n eps s_0; 8 of them are allowed."""
    t = [np.ones((2, 1, 1, 1, 1)) for _ in range(4)]
    g = gpu_ctm(t, [[0, 1], [2, 3]], n)
    rng = np.random.default_rng(n)
    ref = np.zeros((4, 2, 2, n))
    kinds = ["dense", "graded", "sparse", "graded"]
    for j in range(4):
        for y in range(2):
            for x in range(2):
                m = _corner(rng, n, kinds[(j + 2 * y + x) % 4]) * 10.0 ** (5 * j - 7)
                g.set_env(j, x, y, m)
                s = np.linalg.svd(m, compute_uv=False)
                ref[j, y, x] = s / s[0]
    out = g.spectra()
    g.close()
    assert np.all(np.diff(out, axis=-1) <= 0.0)
    assert np.abs(out - ref).max() < 8 * n * EPS


@pytest.mark.parametrize("prec,chi,tol", [("fp64tc", 120, 1e-10), ("bf16x6", 47, 1e-6), ("bf16x6", 120, 1e-6),
                                          ("bf16x6", 242, 1e-6)])
def test_projector_cores_at_wide_rows(prec, chi, tol):
    """Projector cores of k = chi + 16 columns on both sides of the 128 and 256
    element register tiles, cold and (second sweep) from the previous V."""
    cut = 1e-8 if prec == "fp64tc" else 1e-6
    t = [synth.product_plus_noise(6, 0, 4, 2)]
    g = gpu_ctm(t, [[0]], chi, prec=prec, cutoff=cut)
    g.sweep(2)
    st = O.make_state(t, [[0]], 2, chi)
    opt = O.CTMOptions(chi=chi, proj="svd", cutoff=cut)
    for _ in range(2):
        st = O.sweep(st, opt)
    assert np.abs(g.site_rdms() - O.site_rdms(st, t, [[0]])).max() < tol
    g.close()
