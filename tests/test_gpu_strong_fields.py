"""Strong fields on weakly coupled or decoupled sites: factors whose entries span more than
FP64's 53 bits by place, where rounding against a row's or column's largest entry alone
(as digits do) is not enough.  References: fixed-point integers of 640 bits, and closed forms."""
import decimal
import math

import numpy as np
import pytest

import dqmc_inputs as di

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
GTOL, LTOL = 1e-10, 1e-9
P = 640                                     # bits behind the point


@pytest.fixture(scope="module")
def dq():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2003_05286_gb300 as m
    m.lib()
    return m


def _dev(x):
    return torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device="cuda")


def _ising(N, M, lam, seed):
    return lam * (2.0 * np.random.default_rng(seed).integers(0, 2, (M, N)) - 1)


def _ring_greens(t, dtau, V, terms=24):
    """G and log det of a ring with hopping -t: B_l by the Taylor series of the sparse
    exp(-dtau K), G by Gaussian elimination with row pivoting."""
    M, N = V.shape
    decimal.getcontext().prec = 220
    ev = {v: int(decimal.Decimal(v).exp() * (1 << P)) for v in np.unique(V)}
    a = int(decimal.Decimal(t) * decimal.Decimal(dtau) * (1 << P))      # (-dtau K) has a beside the diagonal
    B = np.zeros((N, N), dtype=object)
    for i in range(N):
        B[i, i] = 1 << P
    for l in range(M):
        B = B * np.array([ev[v] for v in V[l]], dtype=object)[:, None] >> P
        term = B
        for n in range(1, terms):
            term = ((np.roll(term, 1, 0) + np.roll(term, -1, 0)) * a >> P) // n
            if not term.any():
                break
            B = B + term
    for i in range(N):
        B[i, i] += 1 << P
    A = np.concatenate([B, np.zeros((N, N), dtype=object)], 1)
    ld = 0.0
    for i in range(N):
        A[i, N + i] = 1 << P
    for i in range(N):
        p = i + max(range(N - i), key=lambda r: abs(A[i + r, i]))
        A[[i, p]] = A[[p, i]]
        piv = A[i, i]
        ld += math.log(abs(piv)) - P * math.log(2.0)
        A[i] = (A[i] << P) // piv
        f = A[:, i].copy()
        f[i] = 0
        A = A - (f[:, None] * A[i][None, :] >> P)
    return (A[:, N:] / (1 << P)).astype(float), ld


@pytest.mark.parametrize("k", [5, 10])
@pytest.mark.parametrize("N,seed", [(100, 10000), (130, 13005)])
def test_tree_of_weakly_coupled_sites(dq, N, seed, k):
    """Row-graded QRs whose pivots D_1 orders, not the columns' norms (hopping 1e-3)."""
    V = _ising(N, 40, 1.2, seed)
    Gx, ldx = _ring_greens(1e-3, 0.1, V)
    G, ld, sg, st = dq.greens(_dev(1e-3 * di.chain_hopping(N)), 0.1, _dev(V), k, handle=dq.Handle(fold=1))
    assert int(st) == 0 and int(sg) == 1
    assert np.abs(G.cpu().numpy() - Gx).max() <= GTOL
    assert abs(float(ld) - ldx) <= LTOL * max(1.0, abs(ldx))


def _sites(kind, N):
    return np.zeros(N) if kind == "alike" else np.linspace(-3.0, 3.0, N)


@pytest.mark.parametrize("k", [5, 10])
@pytest.mark.parametrize("kind", ["alike", "levels"])
@pytest.mark.parametrize("N", [48, 64, 100, 160, 257])
def test_sites_alone(dq, N, kind, k):
    """K diagonal: every site is its own problem, whatever the others' fields (factors e^{+-30}
    of each other in one chunk).  G = 1 / (1 + e^{s}) with s a sum of M terms of order one: a
    few M rounding errors of 2^-53 each."""
    M, K = 40, _sites(kind, N)
    tol = 4 * M * 2.0 ** -53
    V = 2.0 * np.random.default_rng(100 * N).standard_normal((2, M, N))
    sums = V.sum(1) - 0.1 * M * K
    g, h = 1.0 / (1.0 + np.exp(sums)), dq.Handle(fold=0)
    Kd, Vd = _dev(np.diag(K)), _dev(V)
    G, ld, sg, st = dq.greens(Kd, 0.1, Vd, k, handle=h)
    assert int((st != 0).sum()) == 0 and int((sg != 1).sum()) == 0
    G = G.cpu().numpy()
    for b in range(2):
        assert np.abs(G[b] - np.diag(g[b])).max() <= tol
        want = np.log1p(np.exp(sums[b])).sum()
        assert abs(float(ld[b]) - want) <= tol * (1.0 + np.abs(sums[b])).sum()
    _, Gt0, st = dq.greens_tdisplaced(Kd, 0.1, Vd, k, want_tt=False)
    assert int((st != 0).sum()) == 0
    for b in range(2):
        for j in range(Gt0.shape[1]):
            t0 = np.exp(V[b, : j * k].sum(0) - 0.1 * j * k * K) * g[b]
            assert np.abs(Gt0[b, j].cpu().numpy() - np.diag(t0)).max() <= tol * max(1.0, t0.max())


@pytest.mark.parametrize("k", [5, 10])
@pytest.mark.parametrize("N", [64, 160])
def test_sites_alone_tree(dq, N, k):
    """The same in the tree fold, whose factors are graded on both sides; the suite's tolerance."""
    V = np.stack([_ising(N, 40, 1.2, 100 * N + s) for s in range(4)])
    s = V.sum(1)
    G, ld, sg, st = dq.greens(_dev(np.zeros((N, N))), 0.1, _dev(V), k, handle=dq.Handle(fold=1))
    assert int((st != 0).sum()) == 0
    for b in range(4):
        assert np.abs(G[b].cpu().numpy() - np.diag(1.0 / (1.0 + np.exp(s[b])))).max() <= GTOL
        want = np.log1p(np.exp(s[b])).sum()
        assert abs(float(ld[b]) - want) <= LTOL * max(1.0, want)
