"""Setup transform in its prime-factor form (fft_setup.cu): every prime power
and several together, more than one pass per power, series rows that straddle
two rows of Fhat (odd N_m), single columns, host blocks in device memory or
staged; 6480 is past its shared memory (the mixed-radix kernel runs)."""
import numpy as np
import pytest
import torch

import synth
from oracle import fft_method, quantize
import paper_2407_13066_gb300 as btt

pytestmark = pytest.mark.gpu

SHAPES = [  # (N_t, N_d, N_m)
    (1, 2, 3), (2, 1, 1), (7, 3, 5), (16, 4, 6), (27, 1, 9), (49, 5, 3), (125, 2, 4), (360, 3, 7), (512, 1, 3),
    (1125, 2, 3), (2520, 1, 5), (4096, 1, 2), (6480, 1, 3),
]


@pytest.mark.parametrize("shape", SHAPES)
def test_stored_fhat(shape):
    """FP64 storage to 1e-13 of the largest entry (the bound of the 64-step
    test), FP32 to one unit in the last place of it, FP16 scales to 1e-6."""
    N_t, N_d, N_m = shape
    w = synth.Workload("setup", N_t, N_d, N_m, tau=max(1.0, N_t / 5), seed=N_t + N_m)
    F = synth.blocks(w)
    ref = fft_method.setup(F)
    top = np.abs(ref).max()
    for prec, dtype, tol in (("f64", np.complex128, 1e-13), ("f32", np.complex64, 2.0 ** -23)):
        raws = []
        for blocks in (F, torch.from_numpy(F).cuda()):
            with btt.Operator(blocks, precision=prec) as op:
                raw, _ = op.copy_fhat()
                ld = op.fhat_ld()
            raws.append(raw)
        assert np.array_equal(raws[0], raws[1])
        got = raws[0].view(dtype).reshape(N_t + 1, N_d, ld)
        assert np.abs(got[:, :, :N_m] - ref).max() <= tol * top
        assert np.all(got[:, :, N_m:] == 0)
    with btt.Operator(F, precision="f16s") as op:
        _, sc = op.copy_fhat()
    np.testing.assert_allclose(sc, quantize.fp16_scales(ref), rtol=1e-6)


@pytest.mark.parametrize("shape", SHAPES + [(20, 33, 5), (96, 3, 700)])
def test_fp64_vectors(shape):
    """F, F* and the Hessian of two FP64 vectors on the same passes (forward
    halves on their own CTAs, the inverse, the middle step): the FP64 bound."""
    N_t, N_d, N_m = shape
    w = synth.Workload("pf64", N_t, N_d, N_m, tau=max(1.0, N_t / 5), seed=2 * N_t + N_m)
    F, m, d = synth.blocks(w), synth.vectors(w, "m", 2), synth.vectors(w, "d", 2)
    g = synth.noise_gamma_inv(w)
    Fh = fft_method.setup(F)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    rel = lambda a, b: np.linalg.norm(a.cpu().numpy() - b) / np.linalg.norm(b)
    with btt.Operator(dev(F), precision="f64", max_nrhs=2) as op:
        f = fft_method.forward(Fh, m)
        assert rel(op.matvec(dev(m)), f) < 1e-12
        assert rel(op.adjoint(dev(d)), fft_method.adjoint(Fh, d)) < 1e-12
        assert rel(op.hessian(dev(m), dev(g)), fft_method.adjoint(Fh, g * f)) < 1e-12
        assert rel(op.hessian(dev(m)), fft_method.adjoint(Fh, f)) < 1e-12


@pytest.mark.parametrize("prec", ["f16s", "fp8s"])
@pytest.mark.parametrize("shape", [(16, 4, 6), (360, 2, 9), (6480, 1, 3)])
def test_scales_of_a_slice_that_holds_nan(shape, prec):
    """Two NaN samples in neighbouring columns make both columns NaN at every
    frequency; such a slice has no largest magnitude and takes scale 1, from
    the prime-factor kernel as from the mixed-radix one (6480)."""
    N_t, N_d, N_m = shape
    w = synth.Workload("setupnan", N_t, N_d, N_m, tau=N_t / 5, seed=N_t)
    F = synth.blocks(w)
    F[N_t // 3, 0, 0:2] = np.nan
    with btt.Operator(F, precision=prec) as op:
        _, sc = op.copy_fhat()
    np.testing.assert_array_equal(sc, np.ones(N_t + 1))


@pytest.mark.parametrize("shape", [(5250, 1, 4), (5400, 2, 3), (6000, 1, 3), (6400, 1, 2)])
def test_stored_fhat_at_the_largest_tiles(shape):
    """Up to 6456 steps the prime-factor tile fits (with the maxima of the scaled
    formats up to 5282, their pass takes the mixed-radix kernel above), the
    mixed-radix one to 5811 and in global scratch beyond."""
    test_stored_fhat(shape)
