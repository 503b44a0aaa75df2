"""Residue transforms (fft_residue.cu): every cluster size (N_t divisible by
1, 2, 4, 8), no pass to several, every radix, narrow and ragged tiles, rows on
and off 16-byte boundaries, both output and both input formats."""
import numpy as np
import pytest
import torch

import synth
from oracle import fft_method
import paper_2407_13066_gb300 as btt
from tests.test_gpu_parity import TOL, dev, host, inputs

pytestmark = pytest.mark.gpu
rel = lambda a, b: np.linalg.norm(a - b) / np.linalg.norm(b)

SHAPES = [  # (N_t, N_d, N_m)
    (1, 1, 3), (2, 3, 5), (3, 2, 4), (7, 5, 9), (8, 1, 16), (18, 2, 33), (40, 3, 21), (49, 4, 70),
    (105, 1, 5), (343, 2, 8), (420, 7, 45), (720, 3, 64), (1125, 2, 17), (1500, 5, 39), (3000, 2, 12),
    (5000, 1, 10), (6561, 1, 3), (9000, 3, 13), (12288, 1, 6),
]


@pytest.mark.parametrize("shape", SHAPES)
def test_fp32(shape):
    """FP32 against the oracle's FFT algorithm (the only one fast enough here),
    two vectors; the Hessian covers the middle step."""
    N_t, N_d, N_m = shape
    w = synth.Workload("res", N_t, N_d, N_m, tau=max(1.0, N_t / 5), seed=N_t + N_m)
    F, m, d, g = inputs(w, nrhs=2)
    Fh = fft_method.setup(F)
    with btt.Operator(torch.from_numpy(F).cuda(), precision="f32", max_nrhs=2) as op:
        assert rel(host(op.matvec(dev(m, torch.float32))), fft_method.forward(Fh, m)) < TOL["f32"]
        assert rel(host(op.adjoint(dev(d, torch.float32))), fft_method.adjoint(Fh, d)) < TOL["f32"]
        got = host(op.hessian(dev(m, torch.float32), dev(g, torch.float32)))
        op.device_status()
    assert rel(got, fft_method.adjoint(Fh, g * fft_method.forward(Fh, m))) < TOL["f32"]


@pytest.mark.parametrize("prec", ["bf16", "bf16x2"])
@pytest.mark.parametrize("shape", [(40, 5, 21), (105, 3, 9), (420, 6, 36), (1500, 4, 19), (3000, 2, 8), (9000, 2, 5)])
def test_tensor_operands(shape, prec):
    """The BF16 operand (and its remainder plane) and the BF16 inverse input."""
    N_t, N_d, N_m = shape
    w = synth.Workload("restc", N_t, N_d, N_m, tau=N_t / 5, seed=N_t + 3 * N_m)
    F, m, d, _ = inputs(w, nrhs=17)
    Fh = fft_method.setup(F)
    with btt.Operator(torch.from_numpy(F).cuda(), precision=prec, max_nrhs=17, gemm="tensor") as op:
        assert rel(host(op.matvec(dev(m, torch.float32))), fft_method.forward(Fh, m)) < TOL[prec]
        assert rel(host(op.adjoint(dev(d, torch.float32))), fft_method.adjoint(Fh, d)) < TOL[prec]
        op.device_status()


@pytest.mark.parametrize("N_t", [60, 1500])
def test_pointer_table(N_t):
    """Vectors at addresses 4 bytes past a 16-byte boundary give the results
    of the contiguous batch, bit for bit."""
    from paper_2407_13066_gb300 import _lib
    import ctypes
    N_d, N_m, nrhs = 3, 40, 3
    w = synth.Workload("resptr", N_t, N_d, N_m, tau=N_t / 4, seed=N_t)
    F, m, _, g = inputs(w, nrhs=nrhs)
    with btt.Operator(torch.from_numpy(F).cuda(), precision="f32", max_nrhs=nrhs) as op:
        x, gam = dev(m, torch.float32), dev(g, torch.float32)
        ref = host(op.hessian(x, gam))
        n = N_t * N_m
        raw_in = [torch.zeros(n + 4, device="cuda") for _ in range(nrhs)]
        raw_out = [torch.zeros(n + 4, device="cuda") for _ in range(nrhs)]
        for b in range(nrhs):
            raw_in[b][1:n + 1] = x[b].reshape(-1)
        P = ctypes.c_void_p * nrhs
        pin, pout = P(*[t.data_ptr() + 4 for t in raw_in]), P(*[t.data_ptr() + 4 for t in raw_out])
        st = torch.cuda.current_stream().cuda_stream
        _lib.check(op._lib.btt_hessian_batched(op.handle, pin, gam.data_ptr(), pout, nrhs, st))
        torch.cuda.synchronize()
        for b in range(nrhs):
            got = raw_out[b][1:n + 1].double().cpu().numpy().reshape(N_t, N_m)
            np.testing.assert_array_equal(got, ref[b])
            assert raw_out[b][0] == 0 and float(raw_out[b][n + 1:].abs().sum()) == 0


LONG_ODD = [  # (N_t, N_d, N_m): 384 threads per CTA to 2601 steps, 768 above; up to 32 columns the mixed-radix kernels
    (2187, 3, 37), (2401, 33, 6), (2625, 2, 40), (2835, 1, 33), (3125, 2, 36), (3375, 34, 2), (4375, 2, 101),
    (5145, 101, 3), (3125, 1, 20), (5103, 2, 8),
]


@pytest.mark.parametrize("shape", LONG_ODD)
def test_long_odd_lengths(shape):
    """One CTA per tile at its largest sizes, against the oracle's FFT
    algorithm; a vector's bits are the same alone and in a batch of five."""
    N_t, N_d, N_m = shape
    w = synth.Workload("resodd", N_t, N_d, N_m, tau=N_t / 5, seed=N_t + N_m)
    F, m, d, g = inputs(w, nrhs=5)
    Fh = fft_method.setup(F)
    with btt.Operator(torch.from_numpy(F).cuda(), precision="f32", max_nrhs=5) as op:
        m, d, g = (dev(a, torch.float32) for a in (m, d, g))
        for f, x, ref in ((op.matvec, m, fft_method.forward(Fh, host(m))),
                          (op.adjoint, d, fft_method.adjoint(Fh, host(d))),
                          (lambda v: op.hessian(v, g), m,
                           fft_method.adjoint(Fh, host(g) * fft_method.forward(Fh, host(m))))):
            y = f(x)
            assert rel(host(y), ref) < TOL["f32"]
            assert torch.equal(torch.cat([f(x[j:j + 1]) for j in range(5)]), y)
        op.device_status()


@pytest.mark.parametrize("prec", ["bf16", "bf16x2"])
@pytest.mark.parametrize("shape", [(2401, 3, 19), (3125, 2, 35), (5145, 1, 6)])
def test_long_odd_tensor_operands(shape, prec):
    """Their BF16 forms, to the oracle at the format's tolerance."""
    N_t, N_d, N_m = shape
    w = synth.Workload("resoddtc", N_t, N_d, N_m, tau=N_t / 5, seed=N_t + 3 * N_m)
    F, m, d, _ = inputs(w, nrhs=17)
    Fh = fft_method.setup(F)
    with btt.Operator(torch.from_numpy(F).cuda(), precision=prec, max_nrhs=17, gemm="tensor") as op:
        assert rel(host(op.matvec(dev(m, torch.float32))), fft_method.forward(Fh, m)) < TOL[prec]
        assert rel(host(op.adjoint(dev(d, torch.float32))), fft_method.adjoint(Fh, d)) < TOL[prec]
        op.device_status()
