"""Accuracy of the BF16x6 form's FP32 accumulation, in one product whose K is split
and in the RDMs of the case that magnifies it most."""
import numpy as np
import pytest

import synth
from gpu_common import gpu_ctm
from test_gpu_tc_gemm import _zgemm_tile

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bn,splits", [(128, 2), (128, 27), (256, 2), (256, 5), (256, 27)])
@pytest.mark.parametrize("shape", [(848, 69, 848), (130, 100, 53), (1500, 256, 256)])
def test_product_error_is_that_of_one_accumulation_per_k_step(shape, bn, splits):
    """An accumulation on the tensor cores cuts the running sum by half an ulp
    on average (2^-24 to 2^-23 of it; 2^-23 taken), and the running sum of random
    terms has grown to sqrt(j / n) of the result after j of n steps: (1/3) n 2^-23
    of the result for the n = 2K / 16 / splits steps of a run.  2^-23 for the
    operands' 24 bits and the sum of the runs."""
    M, N, K = shape
    rng = np.random.default_rng(M + bn + splits)
    A = rng.standard_normal((M, K)) + 1j * rng.standard_normal((M, K))
    B = rng.standard_normal((K, N)) + 1j * rng.standard_normal((K, N))
    C = _zgemm_tile(3, bn, splits, A, 0, B, 0, M, N, K)
    ref = A @ B
    err = np.linalg.norm(C - ref) / np.linalg.norm(ref)
    blocks = 2 * ((2 * K + 63) // 64)  # k-blocks of two steps, padded to pairs
    steps = 2 * (-(-blocks // min(splits, blocks)))
    print(f"{shape} bn {bn} splits {splits}: {err:.2e}")
    assert err < (steps / 3 + 1) * 2.0 ** -23


def test_two_corner_rdms_of_a_2x1_cell():
    """RDMs of a 2x1 cell at D = 4, chi = 53 with two-corner projectors after three
    sweeps against the FP64-accurate form at the same cutoff, over 16 states: the
    case magnifies the products' rounding by a factor that differs from state to
    state, so the mean is held to a bound.  0.8e-6 lies between the means of one
    accumulator for all six products (1.2e-6) and of two (6e-7), both over 40 other
    states."""
    err = []
    for seed in range(16):
        t = [synth.product_plus_noise(seed, i, 8, 4) for i in range(2)]
        rho = []
        for prec in ("fp64tc", "bf16x6"):
            g = gpu_ctm(t, [[0, 1]], 53, prec=prec, cutoff=1e-6, corners=2)
            g.sweep(3)
            rho.append(g.rdms())
            g.close()
        err.append(max(np.linalg.norm(rho[1][k] - rho[0][k]) / np.linalg.norm(rho[0][k]) for k in ("h", "v")))
    print(f"mean {np.mean(err):.1e} largest {max(err):.1e}")
    assert np.mean(err) < 0.8e-6
