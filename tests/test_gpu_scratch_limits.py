"""Forms whose scratch is too small for what the larger cells keep there: the corners'
digit planes of the FP64-accurate form, the rotation log, the k x k core of plain FP64."""
import numpy as np
import pytest

import oracle as O
import synth
from gpu_common import gpu_ctm, oracle_options, spectra_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,D,chi,prec,budget,corners", [
    (1, 3, 100, "fp64tc", 40, 4),    # planes of 4 x 2 corners do not fit beside the core
    (1, 3, 100, "fp64tc", 40, 2),    # those of 2 x 2 do
    (1, 3, 100, "fp64tc", 9000, 4),  # nor does the rotation log
    (1, 2, 60, "fp64", 64, 4),       # nor does the log of the largest budget with one
    (8, 2, 40, "fp64tc", 40, 4)])    # all of it fits
def test_small_scratch_gives_the_same_results(d, D, chi, prec, budget, corners):
    """One-tensor cell with d physical states after two sweeps: corner spectra and
    one-site RDM against the oracle at the same truncation, 1e-9 (two corners: the
    range finder's distance from the exact SVD, 1e-7)."""
    t = [synth.product_plus_noise(3, 0, d, D)]
    g = gpu_ctm(t, [[0]], chi, prec=prec, jacobi_max_sweeps=budget, corners=corners)
    g.sweep(2)
    st = O.make_state(t, [[0]], D, chi)
    opt = oracle_options(chi, D, corners=corners)
    for _ in range(2):
        st = O.sweep(st, opt)
    tol = 1e-9 if corners == 4 else 1e-7
    assert spectra_err(g.spectra(), O.corner_spectra(st)) < tol
    assert np.abs(g.site_rdms() - O.site_rdms(st, t, [[0]])).max() < tol
    g.close()


@pytest.mark.parametrize("chi", [40, 200])
def test_product_state_without_room_for_the_core(chi):
    """D = 1: K = chi below k = chi + 16; at chi = 200 the k x k factors outgrow the
    scratch and plain FP64 takes one-sided Jacobi on the full rows."""
    rng = np.random.default_rng(chi)
    a = rng.standard_normal((2, 1, 1, 1, 1)) + 1j * rng.standard_normal((2, 1, 1, 1, 1))
    g = gpu_ctm([a], [[0]], chi)
    g.sweep(2)
    v = a.reshape(-1)
    rho = np.outer(v, v.conj()) / np.vdot(v, v).real
    out = g.site_rdms()
    g.close()
    assert min(np.abs(out - rho).max(), np.abs(out - rho.T).max()) < 1e-12
