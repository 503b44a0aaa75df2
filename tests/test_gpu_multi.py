"""Several vectors per pass over Fhat on the FP32 units (gemv_multi.cu): row
groups of 4 and tiles of 32, ragged rows and columns, chunks with tails, warps
that share the columns (few rows), group sizes 2 .. 8 and several groups."""
import numpy as np
import pytest
import torch

import synth
from oracle import direct, fft_method, quantize
import paper_2407_13066_gb300 as btt
from tests.test_gpu_parity import QFMT, TOL, dev, host, inputs

pytestmark = pytest.mark.gpu

SHAPES = [  # (N_t, N_d, N_m)
    (16, 1, 1), (16, 7, 2500), (12, 33, 4099), (10, 130, 513), (160, 37, 4100), (160, 3, 70),
]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("prec", ["f32", "f16s", "bf16", "bf16x2", "fp8s"])
def test_vector_groups(shape, prec):
    """Against the FP64 definition at the format's tolerance, and against the
    oracle's algorithm on the same rounded Fhat, where only FP32 arithmetic
    remains (4e-6, the bound of the single-vector kernels' test)."""
    N_t, N_d, N_m = shape
    w = synth.Workload("multi", N_t, N_d, N_m, tau=N_t / 3, envelope=prec != "f32", seed=N_d * 7 + N_m)
    nmax = 19
    F, m, d, _ = inputs(w, nrhs=nmax)
    fwd, adj = direct.forward(F, m), direct.adjoint(F, d)
    Fq = quantize.quantize(fft_method.setup(F), QFMT[prec])
    fwd_q, adj_q = fft_method.forward(Fq, m), fft_method.adjoint(Fq, d)
    with btt.Operator(F, precision=prec, max_nrhs=nmax, gemm="simt") as op:
        for n in (2, 3, 4, 5, 8, 11, 19):
            dm = host(op.matvec(dev(m[:n], torch.float32)))
            md = host(op.adjoint(dev(d[:n], torch.float32)))
            assert direct.rel_l2(dm, fwd[:n]) < TOL[prec]
            assert direct.rel_l2(md, adj[:n]) < TOL[prec]
            for j in range(n):   # every vector by itself
                assert direct.rel_l2(dm[j], fwd_q[j]) < 4e-6
                assert direct.rel_l2(md[j], adj_q[j]) < 4e-6
        op.device_status()


def test_padding_columns_stay_zero():
    """Columns between N_m and the padded row length are not written by F*:
    a non-finite data vector leaves the next F unharmed."""
    N_t, N_d, N_m = 12, 5, 41
    w = synth.Workload("multipad", N_t, N_d, N_m, tau=4.0, seed=3)
    F, m, d, _ = inputs(w, nrhs=6)
    with btt.Operator(F, precision="f32", max_nrhs=6) as op:
        bad = dev(d, torch.float32)
        bad[2] = float("nan")
        op.adjoint(bad)
        got = host(op.matvec(dev(m, torch.float32)))
    assert direct.rel_l2(got, direct.forward(F, m)) < TOL["f32"]


FULL = [  # (N_t, N_d, N_m): grids of several waves, so that a batch of up to 8 stays one group
    (600, 33, 70), (300, 33, 1100),
]


@pytest.mark.parametrize("shape", FULL)
@pytest.mark.parametrize("prec", ["f32", "f16s", "bf16", "bf16x2", "fp8s"])
def test_whole_groups(shape, prec):
    """The kernels of 5 to 8 vectors (F* of FP8 up to 4; F of split pairs has its
    own there): 601 x 2 tiles of rows are 4 waves of two CTAs per SM, where one pass
    for all vectors costs 4 (n + 1) against 8 (n / 2 + 1) for two halves; F*
    has 601 column tiles of 608 resident.  Every vector against the oracle's
    algorithm on the same rounded Fhat (4e-6, as above)."""
    N_t, N_d, N_m = shape
    w = synth.Workload("groups", N_t, N_d, N_m, tau=N_t / 3, envelope=prec != "f32", seed=N_d * 7 + N_m)
    F, m, d, _ = inputs(w, nrhs=8)
    Fq = quantize.quantize(fft_method.setup(F), QFMT[prec])
    fwd_q, adj_q = fft_method.forward(Fq, m), fft_method.adjoint(Fq, d)
    with btt.Operator(torch.from_numpy(F).cuda(), precision=prec, max_nrhs=8, gemm="simt") as op:
        for n in (2, 3, 4, 5, 6, 7, 8):
            dm = host(op.matvec(dev(m[:n], torch.float32)))
            md = host(op.adjoint(dev(d[:n], torch.float32)))
            for j in range(n):
                assert direct.rel_l2(dm[j], fwd_q[j]) < 4e-6
                assert direct.rel_l2(md[j], adj_q[j]) < 4e-6
        op.device_status()
