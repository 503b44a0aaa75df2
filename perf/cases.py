"""Timed cases: the calls a user of the package makes, over their real range of sizes.

A case names the call (`call`), the storage format and the operator's shape
(N_t time steps, N_d observations, N_m parameters per step, nrhs vectors):

    step     F m, F* d and F* Gamma^-1 F m, one call each
    hessian  F* Gamma^-1 F m
    grad     autograd: d = F m and the gradient F* r it gives for an incoming r
    cg       a fixed number of conjugate-gradient iterations on
             (F* Gamma^-1 F + alpha I) x = b
    setup    an operator built from its blocks on the device, one F m with it
    serve    a burst of Hessian requests to the serving loop over resident operators

Inputs are synthetic: blocks F_k = N(0,1) exp(-k/tau), tau = N_t/5, times a
smooth spatial envelope where the case says so; vectors N(0,1); noise
variances uniform in [0.5, 2].
"""
import math
import random

import torch

import paper_2407_13066_gb300 as btt
from paper_2407_13066_gb300.autograd import apply_F
from paper_2407_13066_gb300.serve import Server

BYTES = {"f64": 16, "f32": 8, "bf16x2": 8, "f16s": 4, "bf16": 4, "fp8s": 2}   # stored Fhat, per entry
SMOOTH_PRIMES = (2, 3, 5, 7)      # factors a transform length may have


def _case(name, call, precision, N_t, N_d, N_m, nrhs=1, **more):
    c = {"name": name, "call": call, "precision": precision, "N_t": N_t, "N_d": N_d, "N_m": N_m, "nrhs": nrhs,
         "gemm": "auto", "envelope": False, "iters": 0}
    c.update(more)
    return c


def listed():
    return [
        # The smallest calls: the operator that is checked against a dense
        # matrix, in the paper's FP64 arithmetic; launches and latency.
        _case("small-f64", "step", "f64", 64, 8, 32),
        # One Hessian action inside somebody's own iterative solver, on the
        # smallest operator of the serving workload.
        _case("solver-f32", "hessian", "f32", 128, 50, 2000),
        # A training step's forward and backward through the map; a length
        # (2 N_t = 840 = 8 3 5 7) and sizes nobody chose for the machine.
        _case("grad-ragged-f32", "grad", "f32", 420, 37, 3001, nrhs=3),
        # The bandwidth workload: F, F* and the Hessian on one vector.
        _case("bandwidth-f32", "step", "f32", 1000, 100, 10000),
        # A long record, few parameters: a shape of the paper's N_t sweep.
        _case("long-f32", "step", "f32", 9000, 100, 800),
        # The precision workload, 24.6 GB of FP16 Fhat, one vector each way.
        _case("precision-f16s", "step", "f16s", 512, 600, 20000, envelope=True),
        # A request of 8 vectors kept at FP32 accuracy on the second serving operator.
        _case("few-rhs-f32", "hessian", "f32", 256, 200, 10000, nrhs=8),
        # A request of 5 vectors in BF16 on few long-record sensors, below the
        # batch size from which the tensor cores are chosen.
        _case("few-rhs-bf16", "hessian", "bf16", 1500, 24, 6000, nrhs=5),
        # The multi-right-hand-side workload: 64 vectors on the tensor cores.
        _case("multi-rhs-bf16", "hessian", "bf16", 256, 200, 50000, nrhs=64),
        # The inverse problem itself: CG on 32 right-hand sides, split pair.
        _case("cg-bf16x2", "cg", "bf16x2", 256, 200, 10000, nrhs=32, iters=6),
        # The setup phase every operator goes through once, from FP64 blocks.
        _case("setup-f32", "setup", "f32", 360, 100, 4000),
        # A burst of requests to the serving loop over three resident operators.
        _case("serve-bf16", "serve", "bf16", 0, 0, 0, nrhs=32, gemm="tensor", requests=18,
              operators="128x50x2000 256x200x10000 1024x100x5000"),
    ]


def _smooth(n):
    """The largest 7-smooth number <= n (the transform takes 2 N_t of that form)."""
    while True:
        m = n
        for p in SMOOTH_PRIMES:
            while m % p == 0:
                m //= p
        if m == 1:
            return n
        n -= 1


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["step", "step", "hessian", "hessian", "hessian", "grad", "cg", "setup"])
    precision = rng.choice(["f32", "f32", "f32", "bf16", "bf16x2", "f16s", "fp8s", "f64"])
    if call == "cg" and precision == "f64":
        precision = "f32"                              # CG takes FP32 vectors
    top = {"setup": 2e8, "cg": 3e8}.get(call, 6e8)     # N_t N_d N_m, within the listed cases' cost
    while True:
        N_t = _smooth(_log_uniform(rng, 40, 7000 if precision == "f64" else 10000))
        N_d = _log_uniform(rng, 5, 600)
        N_m = _log_uniform(rng, 30, 50000)
        size = N_t * N_d * N_m
        if not 1e5 <= size <= top:
            continue
        nrhs = 1 if call == "setup" or rng.random() < 0.35 else _log_uniform(rng, 2, 64)
        if precision == "f64":
            nrhs = min(nrhs, 2)
        # vectors of at most 1 GB, products below those of the largest cases
        if nrhs * N_t * max(N_m, N_d) > 2.5e8 or size * nrhs > (2e9 if precision != "bf16" else 2e10):
            continue
        break
    return {"call": call, "precision": precision, "N_t": N_t, "N_d": N_d, "N_m": N_m, "nrhs": nrhs, "gemm": "auto",
            "envelope": rng.random() < 0.3, "iters": rng.choice([3, 5, 6]) if call == "cg" else 0}


# ------------------------------------------------------------------ inputs
def _dev():
    return torch.device("cuda", torch.cuda.current_device())


def _gen(seed):
    return torch.Generator(device=_dev()).manual_seed(int(seed) % (1 << 62))


def _tau(N_t):
    return N_t / 5.0


def _envelope(n, g):
    """Smooth random factor in [0.1, 1] along one spatial index."""
    u = torch.rand(6, generator=g, device=_dev(), dtype=torch.float64)
    a, phi = 2 * u[:3] - 1, 2 * math.pi * u[3:]
    q = torch.arange(1, 4, device=_dev(), dtype=torch.float64)
    x = torch.arange(n, device=_dev(), dtype=torch.float64) / n
    s = (a[:, None] * torch.cos(2 * math.pi * q[:, None] * x[None, :] + phi[:, None])).sum(0)
    return 0.1 + 0.9 * (0.5 + 0.5 * s / a.abs().sum())


def _blocks(N_t, N_d, N_m, seed, wide, envelope):
    """First block column, float64 [N_t][N_d][N_m] on the GPU, drawn a few
    blocks at a time (normals drawn in FP64 where `wide`, else FP32)."""
    g = _gen(3 * seed + 1)
    env = None
    if envelope:
        env = _envelope(N_d, g)[:, None] * _envelope(N_m, g)[None, :]
    out = torch.empty(N_t, N_d, N_m, dtype=torch.float64, device=_dev())
    decay = torch.exp(-torch.arange(N_t, device=_dev(), dtype=torch.float64) / _tau(N_t))
    step = max(1, (1 << 26) // (N_d * N_m))
    for k in range(0, N_t, step):
        o = out[k:k + step]
        o.copy_(torch.randn(o.shape, generator=g, device=_dev(), dtype=torch.float64 if wide else torch.float32))
        o.mul_(decay[k:k + step, None, None])
        if env is not None:
            o.mul_(env)
    return out


def _vectors(nrhs, N_t, n, dtype, g):
    return torch.randn(nrhs, N_t, n, generator=g, device=_dev(), dtype=dtype)


def _gamma_inv(N_t, N_d, dtype, g):
    return 1.0 / (0.5 + 1.5 * torch.rand(N_t, N_d, generator=g, device=_dev(), dtype=dtype))


def _trace(case):
    """The burst's requests: (operator, vectors) pairs, fixed by the case."""
    rng = random.Random(case["requests"])
    shapes = [tuple(int(v) for v in s.split("x")) for s in case["operators"].split()]
    return shapes, [(rng.randrange(len(shapes)), rng.randint(1, case["nrhs"])) for _ in range(case["requests"])]


def _inputs(case, seed):
    """Everything but the operator: vectors and the noise precision."""
    g = _gen(3 * seed + 2)
    N_t, N_d, N_m, nrhs = case["N_t"], case["N_d"], case["N_m"], case["nrhs"]
    T = torch.float64 if case["precision"] == "f64" else torch.float32
    call = case["call"]
    x = {}
    if call == "serve":
        shapes, reqs = _trace(case)
        x["gamma"] = [_gamma_inv(s[0], s[1], T, g) for s in shapes]
        x["m"] = [_vectors(n, shapes[o][0], shapes[o][2], T, g) for o, n in reqs]
        return x
    x["m"] = _vectors(nrhs, N_t, N_m, T, g)
    if call in ("step", "grad"):
        x["d"] = _vectors(nrhs, N_t, N_d, T, g)
    if call in ("step", "hessian", "cg"):
        x["gamma"] = _gamma_inv(N_t, N_d, T, g)
    if call == "cg":
        # a few per cent of the Hessian's largest eigenvalue, about N_m tau / 2
        x["alpha"] = 0.03 * max(N_m, N_d) * _tau(N_t) / 2
    return x


def prepare(case, seed):
    x = _inputs(case, seed)
    if case["call"] == "serve":
        shapes, _ = _trace(case)
        ops = []
        for i, (N_t, N_d, N_m) in enumerate(shapes):
            ops.append(btt.Operator(_blocks(N_t, N_d, N_m, seed + 1000 * i, False, False), precision=case["precision"],
                                    max_nrhs=case["nrhs"], gemm=case["gemm"], host_staging=0))
        x["y"] = [torch.empty_like(m) for m in x["m"]]
        torch.cuda.synchronize()     # the server's streams read these
        x["server"] = Server(ops, gamma_inv=x["gamma"], pool_bytes=1 << 30, max_batch=case["nrhs"])
        x["case"] = case
        return x
    blocks = _blocks(case["N_t"], case["N_d"], case["N_m"], seed, case["precision"] == "f64", case["envelope"])
    if case["call"] == "setup":
        x["blocks"] = blocks
    else:
        x["op"] = btt.Operator(blocks, precision=case["precision"], max_nrhs=case["nrhs"], gemm=case["gemm"],
                               host_staging=0)
    if case["call"] == "grad" and case["precision"] != "f64":
        x["m"].requires_grad_(True)
    x["case"] = case
    return x


# --------------------------------------------------------------------- run
def run(state):
    case = state["case"]
    call = case["call"]
    if call == "step":
        op = state["op"]
        return [op.matvec(state["m"]), op.adjoint(state["d"]), op.hessian(state["m"], state["gamma"])]
    if call == "hessian":
        return [state["op"].hessian(state["m"], state["gamma"])]
    if call == "grad":
        m = state["m"] if state["m"].requires_grad else state["m"].detach().requires_grad_(True)
        d = apply_F(state["op"], m)
        (grad,) = torch.autograd.grad(d, m, state["d"])
        return [d.detach(), grad]
    if call == "cg":
        x, iterations, _ = state["op"].cg(state["m"], state["alpha"], gamma_inv=state["gamma"],
                                          max_iter=case["iters"], tol=0.0)
        return [x, iterations]
    if call == "setup":
        with btt.Operator(state["blocks"], precision=case["precision"], host_staging=0) as op:
            return [op.matvec(state["m"])]
    _, reqs = _trace(case)
    server = state["server"]
    tickets = [server.submit(o, m, y) for (o, _), m, y in zip(reqs, state["m"], state["y"])]
    for t in tickets:
        server.wait(t)
    return list(state["y"])


# -------------------------------------------------------------------- work
def _action(case, kind, N_t, N_d, N_m, nrhs):
    """(bytes, flops) of one F, F* or Hessian: Fhat read once per pass over
    it (the Hessian's two passes are separated by a transform over all
    frequencies), vectors read and written once; complex products and the
    real transforms of length 2 N_t."""
    real = 8 if case["precision"] == "f64" else 4
    passes = 2 if kind == "H" else 1
    nf, L = N_t + 1, 2 * N_t
    b = passes * nf * N_d * N_m * BYTES[case["precision"]]
    cols = {"F": N_m + N_d, "A": N_m + N_d, "H": 2 * N_m}[kind]
    b += nrhs * N_t * cols * real + (N_t * N_d * real if kind == "H" else 0)
    ncol = {"F": N_m + N_d, "A": N_m + N_d, "H": 2 * N_m + 2 * N_d}[kind]
    f = 8.0 * passes * nf * N_d * N_m * nrhs + 2.5 * L * math.log2(L) * ncol * nrhs
    return b, f


def work(case):
    N_t, N_d, N_m, nrhs = case["N_t"], case["N_d"], case["N_m"], case["nrhs"]
    if case["call"] == "serve":
        shapes, reqs = _trace(case)
        b = f = 0
        for i, s in enumerate(shapes):
            n = sum(v for o, v in reqs if o == i)
            if n:
                # every request of an operator could share the passes over its
                # Fhat up to the batch limit
                batches = -(-n // case["nrhs"])
                bi, fi = _action(case, "H", *s, n)
                b0, _ = _action(case, "H", *s, 0)
                b += bi + (batches - 1) * b0
                f += fi
        return {"bytes": b, "flops": f}
    if case["call"] == "setup":
        b, f = _action(case, "F", N_t, N_d, N_m, nrhs)
        L, cols = 2 * N_t, N_d * N_m
        return {"bytes": b + 8 * N_t * cols + (N_t + 1) * cols * BYTES[case["precision"]],
                "flops": f + 2.5 * L * math.log2(L) * cols}
    if case["call"] == "cg":
        # the first residual and each iteration apply the Hessian once
        b, f = _action(case, "H", N_t, N_d, N_m, 0)
        _, f = _action(case, "H", N_t, N_d, N_m, nrhs)
        n = case["iters"] + 1
        return {"bytes": n * b + 2 * 4 * nrhs * N_t * N_m, "flops": n * f}
    kinds = {"step": "FAH", "hessian": "H", "grad": "FA"}[case["call"]]
    parts = [_action(case, k, N_t, N_d, N_m, nrhs) for k in kinds]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


# ------------------------------------------------------------------- exact
class _Exact:
    """The operator in complex128, a group of observations (rows s) at a
    time; the spectra of the blocks are kept when they are small enough."""

    KEEP = 12 << 30

    def __init__(self, blocks):
        self.blocks = blocks
        self.N_t, self.N_d, self.N_m = blocks.shape
        row = (self.N_t + 1) * self.N_m * 16
        self.rows = max(1, min(self.N_d, (1 << 30) // row))
        self.kept = {} if row * self.N_d <= self.KEEP else None

    def groups(self):
        for s in range(0, self.N_d, self.rows):
            if self.kept is not None and s in self.kept:
                yield s, self.kept[s]
                continue
            fh = torch.fft.rfft(self.blocks[:, s:s + self.rows], n=2 * self.N_t, dim=0)
            if self.kept is not None:
                self.kept[s] = fh
            yield s, fh

    def hat(self, x):
        return torch.fft.rfft(x.double(), n=2 * self.N_t, dim=1)

    def back(self, xh):
        return torch.fft.irfft(xh, n=2 * self.N_t, dim=1)[:, :self.N_t]

    def fwd(self, m):
        mh = self.hat(m).permute(1, 2, 0)                              # [w][l][b]
        dh = [torch.bmm(fh, mh) for _, fh in self.groups()]            # [w][s][b]
        return self.back(torch.cat(dh, 1).permute(2, 0, 1))

    def adj(self, d):
        dh = self.hat(d).permute(1, 2, 0)
        mh = 0
        for s, fh in self.groups():
            mh = mh + torch.bmm(fh.transpose(1, 2).conj(), dh[:, s:s + fh.shape[1]])
        return self.back(mh.permute(2, 0, 1))

    def hess(self, m, gamma):
        return self.adj(self.fwd(m) * gamma.double())


def _exact_cg(op, b, gamma, alpha, iters):
    b = b.double()
    x = torch.zeros_like(b)
    r = b - op.hess(x, gamma) - alpha * x
    p = r.clone()
    rs = (r * r).sum((1, 2), keepdim=True)
    for _ in range(iters):
        hp = op.hess(p, gamma) + alpha * p
        a = rs / (p * hp).sum((1, 2), keepdim=True)
        x = x + a * p
        r = r - a * hp
        new = (r * r).sum((1, 2), keepdim=True)
        p = r + (new / rs) * p
        rs = new
    return x


def exact(case, seed):
    x = _inputs(case, seed)
    call = case["call"]
    if call == "serve":
        shapes, reqs = _trace(case)
        out = [None] * len(reqs)
        for i, s in enumerate(shapes):
            op = _Exact(_blocks(*s, seed + 1000 * i, False, False))
            mine = [j for j, (o, _) in enumerate(reqs) if o == i]
            for j in mine:
                out[j] = op.hess(x["m"][j], x["gamma"][i])
        return out
    op = _Exact(_blocks(case["N_t"], case["N_d"], case["N_m"], seed, case["precision"] == "f64", case["envelope"]))
    if call == "step":
        return [op.fwd(x["m"]), op.adj(x["d"]), op.hess(x["m"], x["gamma"])]
    if call == "hessian":
        return [op.hess(x["m"], x["gamma"])]
    if call == "grad":
        return [op.fwd(x["m"]), op.adj(x["d"])]
    if call == "cg":
        return [_exact_cg(op, x["m"], x["gamma"], x["alpha"], case["iters"]), None]
    return [op.fwd(x["m"])]
