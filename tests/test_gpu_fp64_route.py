"""Plain FP64 projector bases: the CholeskyQR3 route against one-sided Jacobi on
the full rows (which an orth_tol above 1e-14 keeps), both to FP64 results."""
import numpy as np
import pytest

import synth
from gpu_common import gpu_ctm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,chi,pattern,corners,mixed", [
    (1, 40, [[0, 1], [2, 3]], 4, False),   # K = chi below k: rank one
    (2, 8, [[0, 1], [2, 3]], 4, False),    # k = 24: the small-row Jacobi on the core
    (2, 16, [[0]], 4, False), (2, 37, [[0, 1]], 2, False), (3, 20, [[0], [1]], 4, False),
    (3, 27, [[0, 1], [2, 3]], 4, True), (4, 33, [[0, 1], [2, 3]], 2, False)])
def test_cholesky_bases_match_jacobi_bases(D, chi, pattern, corners, mixed):
    nt = len(pattern) * len(pattern[0])
    t = [synth.product_plus_noise(8, i, 4, D) for i in range(nt)]
    bra = [a + 0.02 * synth.product_plus_noise(9, i, 4, D) for i, a in enumerate(t)] if mixed else None
    out = []
    for tol in (1e-14, 1.1e-14):
        g = gpu_ctm(t, pattern, chi, corners=corners, bra=bra, orth_tol=tol)
        g.sweep(3)
        out.append((g.site_rdms(), g.kappa()))
        g.close()
    assert np.abs(out[0][0] - out[1][0]).max() < 1e-10
    assert abs(out[0][1] - out[1][1]) < 1e-10 * abs(out[1][1])


def test_deep_cutoff_and_large_budget_stay_on_the_jacobi_route():
    """A cutoff of 1e-12 (below what a Gram resolves) and a Jacobi budget of
    500 sweeps run as before and agree with the default where it applies."""
    w = synth.workload("real", seed=3, chi=12)
    ref = gpu_ctm(w["tensors"], w["pattern"], 12)
    ref.sweep(4)
    for kw in ({"cutoff": 1e-12}, {"jacobi_max_sweeps": 500}):
        g = gpu_ctm(w["tensors"], w["pattern"], 12, **kw)
        g.sweep(4)
        assert abs(g.energy(w["J"]) - ref.energy(w["J"])) < 1e-8 * abs(ref.energy(w["J"]))
        g.close()
    ref.close()
