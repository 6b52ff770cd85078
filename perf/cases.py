"""Timing cases of the library: the calls a determinant quantum Monte Carlo program makes.

Every case is one pass through the public Python entry points on device
tensors: equal-time Green's functions (one walker or a batch, FP64 or the
tensor-core chain), the log determinant alone, time-displaced functions on the
k-grid, the log determinant with its gradient through autograd, and an uneven
batch replayed as a CUDA graph.  Lattices are periodic squares (L x L, at most
18 x 18) or rings of any length, with the slice width dtau = 0.1 of the
repository's workloads.  The couplings are moderate: a sampler visits fields
with weight |det|, which keeps it away from the nearly singular ones that
independent random fields at strong coupling run into.

``exact`` recomputes a case in 64 bits with plain torch on the host: slices
multiplied in chunks of at most five, each re-factorised by a Householder QR
of the norm-sorted columns, and the D+/D- split inversions.
"""
import concurrent.futures as cf
import math
import os

import torch

import paper_2003_05286_gb300 as dq

DTAU = 0.1


# ---- the cases -------------------------------------------------------------

def listed():
    return [
        # one small walker, eager call: the smallest lattice in use, a sampler
        # re-evaluating G after a sweep; latency and launches are all there is
        dict(name="g16 one", call="greens", lattice="square", L=4, batch=1, M=80, k=10, U=2.0, prec=0),
        # log det alone of one mid-size walker: the weight of a proposed global move
        dict(name="logdet36 one", call="logdet", lattice="square", L=6, batch=1, M=100, k=10, U=2.0, prec=0),
        # one walker on 8 x 8 at low temperature
        dict(name="g64 one", call="greens", lattice="square", L=8, batch=1, M=400, k=10, U=2.0, prec=0),
        # an odd ring, odd chain length (short last chunk), some tens of walkers
        dict(name="g101 odd", call="greens", lattice="ring", L=101, batch=24, M=137, k=7, U=2.0, prec=0),
        # one walker on the largest lattice of the repository's workloads
        dict(name="g256 one", call="greens", lattice="square", L=16, batch=1, M=200, k=10, U=2.0, prec=0),
        # the headline batch: 128 walkers on 16 x 16, beta = 20 (weak coupling, so that none
        # of the many random fields is nearly singular)
        dict(name="g256 batch", call="greens", lattice="square", L=16, batch=128, M=200, k=10, U=1.0, prec=0),
        # the same batch with the tensor-core chain, which a program re-factorises
        # a little more often than the FP64 one
        dict(name="g256 batch bf16x8", call="greens", lattice="square", L=16, batch=128, M=200, k=8, U=1.0, prec=8),
        # above the sizes that are tuned: 18 x 18, a few walkers
        dict(name="g324 few", call="greens", lattice="square", L=18, batch=6, M=60, k=10, U=2.0, prec=0),
        # time-displaced measurements of a batch on 8 x 8, both functions
        dict(name="td64 batch", call="tdisplaced", lattice="square", L=8, batch=256, M=100, k=10, U=2.0, prec=0),
        # the same measurement with the tensor-core chain, all three functions
        dict(name="td64 bf16x8", call="tdisplaced3", lattice="square", L=8, batch=96, M=100, k=5, U=2.0, prec=8),
        # hybrid Monte Carlo force: log det and its gradient, continuous field
        dict(name="grad144 batch", call="grad", lattice="square", L=12, batch=64, M=200, k=10, U=0.0, prec=0),
        # uneven batch in one graph-replayed call: a parallel-tempering run over
        # lattice sizes, temperatures and couplings
        dict(name="ragged", call="ragged", lattice="square", L=16, batch=128, M=400, k=8, U=1.3, prec=0),
    ]


def draw(rng):
    for _ in range(1000):
        c = _draw(rng)
        if c is not None and _cost(c) <= 0.3 * _cost(listed()[5]):
            return c
    raise RuntimeError("no case drawn")


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw(rng):
    call = rng.choice(["greens", "greens", "greens", "logdet", "tdisplaced", "tdisplaced3", "grad", "grad",
                       "ragged"])
    prec = 8 if rng.random() < 0.3 else 0
    if call == "ragged":
        return dict(call=call, lattice="square", L=rng.choice([10, 12, 16]), batch=_log_int(rng, 8, 128),
                    M=rng.randint(100, 400), k=rng.randint(6, 10), U=round(rng.uniform(1.1, 1.5), 2), prec=0)
    lattice = rng.choice(["square", "ring"])
    L = rng.randint(3, 18) if lattice == "square" else _log_int(rng, 12, 320)
    N = L * L if lattice == "square" else L
    if prec and N > 256:
        prec = 0
    displaced = call.startswith("td")
    M = _log_int(rng, 20, 160 if displaced or prec else 400)
    k = rng.randint(4, 6) if prec else rng.randint(5, 10)
    U = 0.0 if call == "grad" else round(rng.uniform(0.8, 1.5), 2)
    return dict(call=call, lattice=lattice, L=L, batch=_log_int(rng, 1, 256), M=M, k=min(k, M), U=U, prec=prec)


# ---- inputs ------------------------------------------------------------------

def _hopping(lattice, L):
    """Nearest-neighbour hopping -1 on the periodic L x L square (site x + L y) or a ring."""
    if lattice == "ring":
        K = torch.zeros(L, L, dtype=torch.float64)
        i = torch.arange(L)
        for a, b in ((i, (i + 1) % L), ((i + 1) % L, i)):
            K[a, b] = -1.0
        return K
    N = L * L
    K = torch.zeros(N, N, dtype=torch.float64)
    s = torch.arange(N)
    x, y = s % L, s // L
    for n in ((x + 1) % L + L * y, (x - 1) % L + L * y, x + L * ((y + 1) % L), x + L * ((y - 1) % L)):
        K[s, n] -= 1.0
    return K


def _field(shape, U, gen, dev):
    """Hirsch field +-lambda (U > 0), or dtau g phi with g = 1.5 and phi ~ N(0, 1) (U = 0)."""
    if U == 0.0:
        return DTAU * 1.5 * torch.randn(shape, dtype=torch.float64, device=dev, generator=gen)
    lam = math.acosh(math.exp(U * DTAU / 2.0))
    return lam * (2.0 * torch.randint(0, 2, shape, device=dev, generator=gen) - 1.0).double()


def _ragged_shapes(case):
    """(L, M, U) of every instance: sizes up to L, M from 100 to M, U from 1 to the case's."""
    sizes = [s for s in (6, 8, 10, 12, 16) if s <= case["L"]]
    out = []
    for i in range(case["batch"]):
        # low-discrepancy fractions: the mix of sizes does not depend on the seed
        a, b, c = (i * 0.7548776662466927) % 1, (i * 0.5698402909980532) % 1, (i * 0.4327254582) % 1
        out.append((sizes[int(a * len(sizes))], 100 + int(b * (case["M"] - 99)), 1.0 + c * (case["U"] - 1.0)))
    return out


def _inputs(case, seed, dev):
    """(K, V) of a uniform case, or the list of (K, V) of a ragged one."""
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    if case["call"] == "ragged":
        Ks = {}
        out = []
        for L, M, U in _ragged_shapes(case):
            if L not in Ks:
                Ks[L] = _hopping("square", L).to(dev)
            out.append((Ks[L], _field((M, L * L), U, gen, dev)))
        return out
    K = _hopping(case["lattice"], case["L"]).to(dev)
    return K, _field((case["batch"], case["M"], K.shape[0]), case["U"], gen, dev)


# A program keeps one handle per setting for its whole run.
_handles = {}


def _handle(prec):
    if prec not in _handles:
        _handles[prec] = dq.Handle(chain_precision=prec)
    return _handles[prec]


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    inputs = _inputs(case, seed, dev)
    if case["call"] == "ragged":
        # the packed batch and the graph-mode handle it is replayed on
        items = [(K, DTAU, V, case["k"]) for K, V in inputs]
        return dict(case=case, batch=dq.RaggedBatch(items), handle=dq.Handle(graphs=True))
    K, V = inputs
    if case["call"] == "grad":
        V.requires_grad_(True)
    return dict(case=case, K=K, V=V, handle=_handle(case["prec"]))


def run(state):
    c = state["case"]
    call, h = c["call"], state["handle"]
    if call == "ragged":
        b = state["batch"]
        _, ld, sg, _ = b.run(h)
        return dict(G=b.Gp, logdet=ld, sign=sg)
    K, V, k = state["K"], state["V"], c["k"]
    if call == "greens":
        G, ld, sg, _ = dq.greens(K, DTAU, V, k, handle=h)
        return dict(G=G, logdet=ld, sign=sg)
    if call == "logdet":
        ld, sg, _ = dq.logdet(K, DTAU, V, k, handle=h)
        return dict(logdet=ld, sign=sg)
    if call == "tdisplaced":
        Gtt, Gt0, _ = dq.greens_tdisplaced(K, DTAU, V, k, handle=h)
        return dict(Gtt=Gtt, Gt0=Gt0)
    if call == "tdisplaced3":
        Gtt, Gt0, G0t, _ = dq.greens_tdisplaced(K, DTAU, V, k, handle=h, want_0t=True)
        return dict(Gtt=Gtt, Gt0=Gt0, G0t=G0t)
    ld = dq.LogDet.apply(V, K, DTAU, k, h)
    (dV,) = torch.autograd.grad(ld.sum(), V)
    return dict(logdet=ld.detach(), dV=dV)


# ---- what a pass cannot do without ---------------------------------------------

def _flops(call, N, M, k):
    nc = -(-M // k)
    chain = 2.0 * M + nc * (8.0 / 3.0 + 1.0)          # slice products, QR with Q, X update
    lu = 2.0 / 3.0
    if call in ("greens", "ragged"):
        return (chain + 2 * (lu + 2.0)) * N ** 3
    if call == "logdet":
        return (chain + 2 * lu + 2.0) * N ** 3
    if call == "tdisplaced":
        return (2 * chain + (nc + 1) * (4 + lu + 4 + 4)) * N ** 3
    if call == "tdisplaced3":
        return (2 * chain + (nc + 1) * (4 + lu + 4 + 6)) * N ** 3
    return (2 * chain + (nc + 1) * (4 + lu + 2 + 2) + (nc + 1) * (k - 1) * 4) * N ** 3


def _sites(case):
    return case["L"] ** 2 if case["lattice"] == "square" else case["L"]


def _cost(case):
    # above 256 sites a walker's factorisations are one after another on one SM each
    return work(case)["flops"] * (8.0 if _sites(case) > 256 else 1.0)


def work(case):
    call, k = case["call"], case["k"]
    if call == "ragged":
        shapes = _ragged_shapes(case)
        Ns = {L * L for L, _, _ in shapes}
        return {"bytes": 8.0 * (sum(n * n for n in Ns) + sum(L * L * M + L ** 4 + 2 for L, M, _ in shapes)),
                "flops": sum(_flops(call, L * L, M, k) for L, M, _ in shapes)}
    N, M, B = _sites(case), case["M"], case["batch"]
    nt = -(-M // k) + 1
    out = {"greens": N * N, "logdet": 0, "tdisplaced": 2 * nt * N * N, "tdisplaced3": 3 * nt * N * N,
           "grad": M * N}[call]
    return {"bytes": 8.0 * (N * N + B * (M * N + out + 2)), "flops": B * _flops(call, N, M, k)}


# ---- the same in 64 bits with plain torch ------------------------------------------

def _udt(A, D):
    """A diag(D) = U diag(D') T by the Householder QR of the norm-sorted columns."""
    key = torch.log(D) + 0.5 * torch.log((A * A).sum(-2))
    p = torch.argsort(key, dim=-1, descending=True)
    q, r = torch.linalg.qr(torch.gather(A, -1, p[:, None, :].expand_as(A)))
    d = torch.diagonal(r, dim1=-2, dim2=-1).abs()
    Dp = torch.gather(D, -1, p)
    t = r / d[..., None] * (Dp[:, None, :] / Dp[..., None])
    T = torch.empty_like(t)
    T.scatter_(-1, p[:, None, :].expand_as(t), t)
    return q, d * Dp, T


def _chain(E, ev, step, cuts, transposed=False):
    """U, D, T of the product of the slices up to each cut (chunks of at most ``step`` slices)."""
    B, M, N = ev.shape
    eye = torch.eye(N, dtype=torch.float64).expand(B, N, N).clone()
    U, D, T = eye, torch.ones(B, N, dtype=torch.float64), eye.clone()
    out = {0: (U, D, T)} if 0 in cuts else {}
    l = 0
    for stop in sorted(c for c in cuts if c > 0):
        while l < stop:
            n = min(l + step, stop)
            A = U
            for s in range(l, n):
                # B_l = E diag(e^{V_l}) from the left, or B_{M-s}^T = diag(e^V) E
                A = ev[:, M - 1 - s, :, None] * (E @ A) if transposed else E @ (ev[:, s, :, None] * A)
            U, D, t = _udt(A, D)
            T = t @ T
            l = n
        out[stop] = (U, D, T)
    return out


def _equal_time(U, D, T, want_G=True):
    Dp, Dm = D.clamp(min=1.0), D.clamp(max=1.0)
    Y = torch.linalg.solve(T, torch.diag_embed(1.0 / Dp))
    Mx = Y + U * Dm[:, None, :]
    sg, lad = torch.linalg.slogdet(Mx)
    sT, _ = torch.linalg.slogdet(T)
    G = torch.linalg.solve(Mx.transpose(-1, -2), Y.transpose(-1, -2)).transpose(-1, -2) if want_G else None
    return G, torch.log(Dp).sum(-1) + lad, (sg * sT).to(torch.int32)


def _displaced(f, b):
    """G(tau,tau), G(tau,0), G(0,tau) from B(tau,0) = U a X and B(beta,tau)^T = W b T."""
    U, a, X = f
    W, c, T = b
    ap, am, bp, bm = a.clamp(min=1.0), a.clamp(max=1.0), c.clamp(min=1.0), c.clamp(max=1.0)
    mid = (U.transpose(-1, -2) @ W) / ap[..., None] / bp[:, None, :] \
        + am[..., None] * (X @ T.transpose(-1, -2)) * bm[:, None, :]
    Z = torch.linalg.solve(mid, torch.cat((U.transpose(-1, -2) / ap[..., None], am[..., None] * X), -1))
    Zt, Z0 = Z.split(U.shape[-1], -1)
    return (W / bp[:, None, :]) @ Zt, (W / bp[:, None, :]) @ Z0, -(T.transpose(-1, -2) * bm[:, None, :]) @ Zt


def _exact_part(call, K, V, k):
    torch.set_num_threads(1)
    E = torch.matrix_exp(-DTAU * K)
    ev = torch.exp(V)
    M = V.shape[1]
    step = min(k, 5)
    if call in ("greens", "logdet", "ragged"):
        return _equal_time(*_chain(E, ev, step, {M})[M], want_G=call != "logdet")
    grid = [min(j * k, M) for j in range(-(-M // k) + 1)] if call != "grad" else \
        sorted(set(range(0, M, step)))
    f = _chain(E, ev, step, set(grid))
    b = _chain(E, ev, step, {M - g for g in grid}, transposed=True)
    if call != "grad":
        pts = [_displaced(f[g], b[M - g]) for g in grid]
        return tuple(torch.stack(x, 1) for x in zip(*pts))
    # gradient: 1 - G_l(i,i), G_{l+1} = B_l G_l B_l^{-1} between the grid points
    _, ld, _ = _equal_time(*_chain(E, ev, step, {M})[M], want_G=False)
    Ei = torch.matrix_exp(DTAU * K)
    dV = torch.empty_like(V)
    for g in grid:
        G = _displaced(f[g], b[M - g])[0]
        for l in range(g, min(g + step, M)):
            dV[:, l] = 1.0 - torch.diagonal(G, dim1=-2, dim2=-1)
            G = E @ (ev[:, l, :, None] * G / ev[:, l, None, :]) @ Ei
    return ld, dV


def exact(case, seed):
    inputs = _inputs(case, seed, torch.device("cuda", torch.cuda.current_device()))
    call, k = case["call"], case["k"]
    if call == "ragged":
        parts = [(K.cpu(), V.cpu()[None]) for K, V in inputs]
    else:
        K, V = inputs[0].cpu(), inputs[1].cpu()
        cores = os.cpu_count() or 1
        parts = [(K, v) for v in V.split(max(1, -(-V.shape[0] // (4 * cores))))]
    threads = torch.get_num_threads()
    with cf.ThreadPoolExecutor(os.cpu_count() or 1) as ex:
        got = list(ex.map(lambda p: _exact_part(call, p[0], p[1], k), parts))
    torch.set_num_threads(threads)
    if call == "ragged":
        return dict(G=torch.cat([g[0].reshape(-1) for g in got]), logdet=torch.cat([g[1] for g in got]),
                    sign=torch.cat([g[2] for g in got]))
    cat = [torch.cat(x) if x[0] is not None else None for x in zip(*got)]
    if call == "greens":
        return dict(G=cat[0], logdet=cat[1], sign=cat[2])
    if call == "logdet":
        return dict(logdet=cat[1], sign=cat[2])
    if call == "tdisplaced":
        return dict(Gtt=cat[0], Gt0=cat[1])
    if call == "tdisplaced3":
        return dict(Gtt=cat[0], Gt0=cat[1], G0t=cat[2])
    return dict(logdet=cat[0], dV=cat[1])
