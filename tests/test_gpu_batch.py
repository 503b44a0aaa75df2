"""On the FP32 and FP64 units a vector's results are the same bits alone and in
any batch: the order in which a row of F is summed depends on the operator's
shape only, and F* and the transforms work on each vector by itself."""
import numpy as np
import pytest
import torch

import synth
import paper_2407_13066_gb300 as btt
from tests.test_gpu_parity import dev, inputs

pytestmark = pytest.mark.gpu

SHAPES = [  # (N_t, N_d, N_m): few rows, few frequencies, both, neither; rows of one block of columns and of many
    (64, 10, 200), (16, 1, 1), (16, 7, 2500), (12, 33, 4099), (160, 3, 70), (64, 8, 2000), (600, 7, 300),
    (160, 37, 4100), (300, 33, 130), (100, 4, 1400), (40, 30, 600),
]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("prec", ["f32", "f16s", "bf16", "bf16x2", "fp8s", "f64"])
def test_same_bits_in_any_batch(shape, prec):
    N_t, N_d, N_m = shape
    w = synth.Workload("inv", N_t, N_d, N_m, tau=N_t / 4, seed=N_t + N_d + N_m)
    nmax = 20
    F, m, d, g = inputs(w, nrhs=nmax)
    m, d, g = (dev(a, torch.float64 if prec == "f64" else torch.float32) for a in (m, d, g))
    with btt.Operator(torch.from_numpy(F).cuda(), precision=prec, max_nrhs=nmax, gemm="simt") as op:
        alone = [torch.cat([f(x[j:j + 1]) for j in range(nmax)])
                 for f, x in ((op.matvec, m), (op.adjoint, d), (lambda v: op.hessian(v, g), m))]
        for n in (2, 3, 4, 6, 8, 11, 20):
            for a, got in zip(alone, (op.matvec(m[:n]), op.adjoint(d[:n]), op.hessian(m[:n], g))):
                assert torch.equal(got, a[:n])
        op.device_status()
