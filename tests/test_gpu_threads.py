"""Operators driven by two host threads at once (each operator by one thread):
what a launch sets on a kernel belongs to the context, not to the operator."""
import threading

import numpy as np
import pytest
import torch

import synth
from oracle import fft_method
import paper_2407_13066_gb300 as btt
from paper_2407_13066_gb300 import _lib
from tests.test_gpu_parity import TOL, dev, host, inputs

pytestmark = pytest.mark.gpu
rel = lambda a, b: np.linalg.norm(a - b) / np.linalg.norm(b)


def drive(calls, n):
    """Every call of `calls` n times in a thread of its own; the statuses that were not OK."""
    bad = [[] for _ in calls]
    gate = threading.Barrier(len(calls))

    def work(i):
        gate.wait()
        for _ in range(n):
            st = calls[i]()
            if st != _lib.BTT_OK:
                bad[i].append(st)

    ts = [threading.Thread(target=work, args=(i,)) for i in range(len(calls))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize()
    return sum(bad, [])


@pytest.mark.parametrize("prec,nrhs,shapes", [
    # F of 8 vectors: 64 and 56 KB of shared memory
    ("f32", 8, [(600, 33, 450), (600, 33, 430)]),
    ("bf16", 8, [(600, 33, 640), (600, 33, 300)]),
    # F of few rows: 64 and 50 KB
    ("fp8s", 2, [(60, 3, 2048), (60, 3, 1600)]),
    # F* of one vector and two: N_d values of dhat each
    ("f32", 2, [(4, 5000, 16), (4, 3200, 16)]),
    ("f16s", 1, [(4, 9000, 16), (4, 6200, 16)]),
])
def test_two_threads(prec, nrhs, shapes):
    calls, keep, checks = [], [], []
    for i, (N_t, N_d, N_m) in enumerate(shapes):
        w = synth.Workload("thr%d" % i, N_t, N_d, N_m, tau=max(1.0, N_t / 5), seed=N_m)
        F, m, d, _ = inputs(w, nrhs=nrhs)
        op = btt.Operator(torch.from_numpy(F).cuda(), precision=prec, max_nrhs=nrhs, gemm="simt")
        st = torch.cuda.Stream()
        x, r = dev(m, torch.float32), dev(d, torch.float32)
        y, z = torch.empty_like(r), torch.empty_like(x)
        keep.append((op, st, x, r, y, z))
        checks.append((fft_method.setup(F), m, d))

        def call(op=op, st=st, x=x, r=r, y=y, z=z):
            a = op._lib.btt_matvec(op.handle, x.data_ptr(), y.data_ptr(), nrhs, st.cuda_stream)
            b = op._lib.btt_adjoint(op.handle, r.data_ptr(), z.data_ptr(), nrhs, st.cuda_stream)
            return a or b
        calls.append(call)
    torch.cuda.synchronize()
    assert drive(calls, 3000) == []
    for (op, _, _, _, y, z), (Fh, m, d) in zip(keep, checks):
        assert rel(host(y), fft_method.forward(Fh, m)) < TOL[prec]
        assert rel(host(z), fft_method.adjoint(Fh, d)) < TOL[prec]
        op.close()
