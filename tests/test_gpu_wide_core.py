"""Projector cores too wide for V beside the rows of a cluster."""
import numpy as np
import pytest

import synth
from gpu_common import gpu_ctm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chi", [288, 304, 310])
def test_double_float_core_with_replayed_v(chi):
    """k = chi + 16 of 304 and 320 (V beside the double-float rows of 16 CTAs) and 326
    (rotations logged and replayed): the RDMs of two sweeps, cold and from the
    previous V, against the FP64-accurate form at the same cutoff, to the form's 1e-6."""
    t = [synth.product_plus_noise(6, 0, 4, 2)]
    rho = []
    for prec in ("fp64tc", "bf16x6"):
        g = gpu_ctm(t, [[0]], chi, prec=prec, cutoff=1e-6)
        g.sweep(2)
        rho.append(g.site_rdms())
        g.close()
    assert np.abs(rho[1] - rho[0]).max() < 1e-6
