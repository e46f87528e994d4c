"""Plain FP64 projector bases: the CholeskyQR3 route against one-sided Jacobi on
the full rows (which an orth_tol above 1e-14 keeps), both to FP64 results.

What FP64 rounding does to the range finder's results depends on the network: a
change of the tensors by 1e-15 moves the one-site RDMs by 1e-15 where the ring's
spectrum falls fast, and by 3e-8 in the two-corner case at D = 4 (LAPACK's
arithmetic does the same to the oracle's range finder; the last basis vectors
carry eps s_0 / s_k of the first, which 1 / s_k in the projectors magnifies).
So the routes may differ by what such a change does to the Jacobi route, times
30 for the roundings of three sweeps."""
import numpy as np
import pytest

import synth
from gpu_common import gpu_ctm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,chi,pattern,corners,mixed", [
    (1, 40, [[0, 1], [2, 3]], 4, False),   # K = chi below k: rank one
    (2, 8, [[0, 1], [2, 3]], 4, False),    # k = 24: the small-row Jacobi on the core
    (2, 16, [[0]], 4, False), (2, 23, [[0]], 4, False), (2, 24, [[0]], 4, False), (2, 25, [[0]], 4, False),
    (2, 37, [[0, 1]], 2, False), (3, 20, [[0], [1]], 4, False),
    (3, 27, [[0, 1], [2, 3]], 4, True), (4, 33, [[0, 1], [2, 3]], 2, False)])
def test_cholesky_bases_match_jacobi_bases(D, chi, pattern, corners, mixed):
    nt = len(pattern) * len(pattern[0])
    t = [synth.product_plus_noise(8, i, 4, D) for i in range(nt)]
    bra = [a + 0.02 * synth.product_plus_noise(9, i, 4, D) for i, a in enumerate(t)] if mixed else None
    rng = np.random.default_rng(chi)
    near = [a * (1.0 + 1e-15 * rng.standard_normal(a.shape)) for a in t]

    def site_rdms(tensors, orth_tol):
        g = gpu_ctm(tensors, pattern, chi, corners=corners, bra=bra, orth_tol=orth_tol)
        g.sweep(3)
        out = g.site_rdms()
        g.close()
        return out

    jacobi = site_rdms(t, 1.1e-14)
    rounding = np.abs(site_rdms(near, 1.1e-14) - jacobi).max()
    assert np.abs(site_rdms(t, 1e-14) - jacobi).max() < 1e-12 + 30 * rounding


@pytest.mark.parametrize("kw", [{"cutoff": 1e-12}, {"jacobi_max_sweeps": 500}])
def test_deep_cutoff_and_large_budget_stay_on_the_jacobi_route(kw):
    """A cutoff of 1e-12 (below what a Gram resolves) and a Jacobi budget beyond
    the rotation log's still run: the same network to the weight of what the
    cutoffs keep or drop and of the noise they amplify (1e-8 and 1e-12 of s_0,
    under s^-1/2 on both sides)."""
    w = synth.workload("real", seed=3, chi=12)
    rho = []
    for k in ({}, kw):
        g = gpu_ctm(w["tensors"], w["pattern"], 12, **k)
        g.sweep(4)
        rho.append(g.site_rdms())
        g.close()
    assert np.isfinite(rho[1]).all() and np.abs(rho[1] - rho[0]).max() < 1e-4
