"""FP64 products on the tensor cores (N >= 64): edges of the 128 x 64 tiles and of
the exact accumulation windows (128 and 256 values of k), both chain directions,
shared and per-instance operands, ended chains, wide and non-finite fields.

The tolerances are the suite's: 1e-10 of max(1, max|G|) in G and 1e-9 relative in
log det against the FP64 oracle, which a product with K 2^-58 of (row max x
column max) per entry stays far below."""
import numpy as np
import pytest

import dqmc_inputs as di
from oracle import dqmc as od

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
GTOL, LTOL = 1e-10, 1e-9


@pytest.fixture(scope="module")
def dq():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2003_05286_gb300 as m
    m.lib()
    return m


def _dev(x):
    return torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device="cuda")


def _field(seed, M, N, amp):
    return amp * di.ising_field(seed, M, N)


def _check(G, ld, sg, K, dtau, V, k):
    Go, ldo, so = od.greens(K, dtau, V, k)
    assert np.abs(G - Go).max() <= GTOL * max(1.0, np.abs(Go).max())
    assert abs(ld - ldo) <= LTOL * max(1.0, abs(ldo)) and sg == so


@pytest.mark.parametrize("fold", [0, 1])
@pytest.mark.parametrize("N", [64, 65, 96, 127, 128, 129, 191, 255, 257, 385])
def test_greens_tile_edges(dq, N, fold):
    K = di.chain_hopping(N)
    V = np.stack([_field(4000 + N + b, 12, N, 0.3) for b in range(2)])
    h = dq.Handle(fold=fold)
    G, ld, sg, st = dq.greens(_dev(K), 0.1, _dev(V), 5, handle=h)
    assert int((st != 0).sum()) == 0
    for b in range(2):
        _check(G[b].cpu().numpy(), float(ld[b]), int(sg[b]), K, 0.1, V[b], 5)


@pytest.mark.parametrize("N", [64, 130])
def test_displaced_and_gradient(dq, N):
    K = di.chain_hopping(N)
    V = _field(4100 + N, 11, N, 0.3)
    Gtt, Gt0, G0t, st = dq.greens_tdisplaced(_dev(K), 0.1, _dev(V), 4, want_0t=True)
    assert int(st) == 0
    Ott, Ot0 = od.greens_tdisplaced(K, 0.1, V, 4)
    for j, l in enumerate(od.tau_grid(11, 4)):
        O0t = od.greens_displaced_back(K, 0.1, V, 4, 0, l)
        for got, want in ((Gtt[j], Ott[j]), (Gt0[j], Ot0[j]), (G0t[j], O0t)):
            assert np.abs(got.cpu().numpy() - want).max() <= GTOL * max(1.0, np.abs(want).max())
    ld, sg, dV, st = dq.logdet_grad(_dev(K), 0.1, _dev(V), 4)
    assert int(st) == 0
    assert np.abs(dV.cpu().numpy() - od.logdet_grad(K, 0.1, V, 4)).max() <= 1e-9


def test_ended_chains(dq):
    """Instances of one group with different M: ended chains pass their product through."""
    N = 72
    K = _dev(di.chain_hopping(N))
    Vs = [_field(4200 + M, M, N, 0.3) for M in (3, 8, 10, 17)]
    Gs, ld, sg, st = dq.greens_ragged([(K, 0.1, _dev(V), 3) for V in Vs])
    assert int((st != 0).sum()) == 0
    for i, V in enumerate(Vs):
        _check(Gs[i].cpu().numpy(), float(ld[i]), int(sg[i]), di.chain_hopping(N), 0.1, V, 3)


def test_wide_entries(dq):
    """Diagonals e^{+-2}: rows and columns of the slices spread over e^4 and more."""
    N = 80
    K, V = di.chain_hopping(N), _field(4300, 6, N, 2.0)
    G, ld, sg, st = dq.greens(_dev(K), 0.1, _dev(V), 1, handle=dq.Handle(fold=0))
    assert int(st) == 0
    _check(G.cpu().numpy(), float(ld), int(sg), K, 0.1, V, 1)


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_non_finite_field(dq, value):
    """A non-finite field entry is flagged for its instance and leaves the other one alone."""
    N = 64
    K = di.chain_hopping(N)
    V = np.stack([_field(4400 + b, 8, N, 0.3) for b in range(2)])
    bad = V.copy()
    bad[1, 3, 7] = value
    h = dq.Handle(fold=0)
    G, ld, sg, st = dq.greens(_dev(K), 0.1, _dev(bad), 4, handle=h)
    assert int(st[0]) == 0 and int(st[1]) != 0
    _check(G[0].cpu().numpy(), float(ld[0]), int(sg[0]), K, 0.1, V[0], 4)
    assert not bool(torch.isfinite(G[1]).all())


def test_without_room_for_digits(dq):
    """Under a memory cap with no room for the digits the products run on the FP64 pipe."""
    N = 64
    K, V = _dev(di.chain_hopping(N)), _dev(np.stack([_field(4500 + b, 8, N, 0.3) for b in range(3)]))
    ref = dq.greens(K, 0.1, V, 4, handle=dq.Handle(fold=0))
    free = dq.Handle(fold=0)
    dq.greens(K, 0.1, V, 4, handle=free)
    for graphs in (False, True):
        h = dq.Handle(fold=0, graphs=graphs)
        h.set_memory_limit(free.device_bytes * 8 // 9 - 3 * 8 * N * N * 8)
        for _ in range(2):
            G, ld, sg, st = dq.greens(K, 0.1, V, 4, handle=h)
            assert (G - ref[0]).abs().max().item() <= GTOL and int((st != 0).sum()) == 0
