"""Plain FP64 truncations outside the Gram route (a cutoff below 1e-9): the
Jacobi SVD of W with its V."""
import numpy as np
import pytest

import oracle as O
import synth
from gpu_common import gpu_ctm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,chi,budget", [(2, 16, 40), (2, 37, 40), (3, 27, 500)])
def test_svd_of_w_stays_on_the_cluster(D, chi, budget):
    """With V beside the rows where both fit a cluster's shared memory, no grid
    barrier is met: a wait limit of one clock cycle, which every wait of the
    grid-barrier kernel runs out of (tests/test_gpu_faults.py), does not show.
    The one-site RDMs against the oracle at the same cutoff."""
    t = [synth.product_plus_noise(5, 0, 8, D)]
    g = gpu_ctm(t, [[0]], chi, cutoff=1e-12, wait_cycles=1, jacobi_max_sweeps=budget)
    g.sweep(2)
    rho = g.site_rdms()
    g.close()
    st = O.make_state(t, [[0]], D, chi)
    opt = O.CTMOptions(chi=chi, proj="svd", cutoff=1e-12)
    for _ in range(2):
        st = O.sweep(st, opt)
    assert np.abs(rho - O.site_rdms(st, t, [[0]])).max() < 1e-10
