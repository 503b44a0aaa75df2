"""Tensor-core products with fewer vectors than a 64-vector tile holds: stages
load the vectors rounded up to 16 rows (F) or 32 rows (F*); the split pair's
forward packs up to 32 vectors into a third stage."""
import numpy as np
import pytest
import torch

import synth
from oracle import direct
import paper_2407_13066_gb300 as btt
from tests.test_gpu_parity import TOL, dev, host, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["bf16", "bf16x2"])
@pytest.mark.parametrize("shape", [(16, 5, 40), (16, 70, 333), (12, 230, 700)])
def test_partial_vector_tiles(shape, prec):
    """Every count of 16-row boxes, one and two tiles, row tiles that leave
    room for the third stage (5, 70) and that do not (230); each after a batch
    whose other vectors are NaN, which must not reach the results."""
    N_t, N_d, N_m = shape
    w = synth.Workload("rows", N_t, N_d, N_m, tau=N_t / 3, seed=N_d + N_m)
    nmax = 97
    F, m, d, _ = inputs(w, nrhs=nmax)
    fwd, adj = direct.forward(F, m), direct.adjoint(F, d)
    bad_m, bad_d = dev(m, torch.float32), dev(d, torch.float32)
    bad_m[1:] = float("nan")
    bad_d[1:] = float("nan")
    with btt.Operator(torch.from_numpy(F).cuda(), precision=prec, max_nrhs=nmax, gemm="tensor") as op:
        for n in (1, 16, 17, 32, 33, 48, 64, 65, 97):
            op.matvec(bad_m)
            op.adjoint(bad_d)
            dm = host(op.matvec(dev(m[:n], torch.float32)))
            md = host(op.adjoint(dev(d[:n], torch.float32)))
            assert direct.rel_l2(dm, fwd[:n]) < TOL[prec]
            assert direct.rel_l2(md, adj[:n]) < TOL[prec]
        op.device_status()
