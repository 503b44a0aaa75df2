"""FP64 F on two and on eight warps per CTA: either side of the lines between
them (152 and 304 CTAs, rows of 64, 512 and 1400 entries), against the oracle."""
import numpy as np
import pytest
import torch

import synth
from oracle import fft_method
import paper_2407_13066_gb300 as btt
from tests.test_gpu_parity import TOL

pytestmark = pytest.mark.gpu

SHAPES = [  # (N_t, N_d, N_m): 9 x 2, 25, 151, 161, 301, 316 and 76 x 4 CTAs
    (8, 7, 1347), (24, 1, 3958), (150, 3, 64), (150, 3, 65), (150, 3, 512), (160, 4, 512), (160, 4, 513), (300, 2, 512),
    (300, 2, 513), (315, 2, 1400), (315, 2, 1401), (75, 13, 1399), (1, 1, 1),
]


@pytest.mark.parametrize("shape", SHAPES)
def test_forward(shape):
    N_t, N_d, N_m = shape
    w = synth.Workload("f64rows", N_t, N_d, N_m, tau=max(1.0, N_t / 5), seed=N_t + N_m)
    F, m = synth.blocks(w), synth.vectors(w, "m", 3)
    ref = fft_method.forward(fft_method.setup(F), m)
    with btt.Operator(torch.from_numpy(F).cuda(), precision="f64", max_nrhs=3) as op:
        y = op.matvec(torch.from_numpy(np.ascontiguousarray(m)).cuda()).cpu().numpy()
    assert np.linalg.norm(y - ref) / np.linalg.norm(ref) < TOL["f64"]
