"""Products with a shared operand on stacked tensor-core tiles: 32-row groups of
several instances in one 128-row tile, ragged last tiles, ended chains inside a
tile, both orientations (E X and X E^{-1}) and the row scale of the backward chain.

The tolerances are the suite's: 1e-10 of max(1, max|G|) in G, 1e-9 in log det
(relative) and in the gradient, against the FP64 oracle, which a product with
K 2^-58 of (row max x column max) per entry stays far below."""
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


def _hopping(N):
    return di.chain_hopping(N) + np.diag(0.2 * np.cos(np.arange(N)))


@pytest.mark.parametrize("N,batch", [(129, 1), (144, 3), (160, 5), (161, 2), (257, 3)])
def test_greens(dq, N, batch):
    K = _hopping(N)
    V = np.stack([0.3 * di.ising_field(6000 + N + b, 7, N) for b in range(batch)])
    G, ld, sg, st = dq.greens(_dev(K), 0.1, _dev(V), 3, handle=dq.Handle(fold=0))
    assert int((st != 0).sum()) == 0
    for b in range(batch):
        Go, ldo, so = od.greens(K, 0.1, V[b], 3)
        assert np.abs(G[b].cpu().numpy() - Go).max() <= GTOL * max(1.0, np.abs(Go).max())
        assert abs(float(ld[b]) - ldo) <= LTOL * max(1.0, abs(ldo)) and int(sg[b]) == so


@pytest.mark.parametrize("N", [64, 81, 144])
def test_gradient_and_every_tau(dq, N):
    K = _hopping(N)
    V = np.stack([0.3 * di.ising_field(6200 + N + b, 7, N) for b in range(3)])
    ld, sg, dV, st = dq.logdet_grad(_dev(K), 0.1, _dev(V), 3)
    assert int((st != 0).sum()) == 0
    for b in range(3):
        assert np.abs(dV[b].cpu().numpy() - od.logdet_grad(K, 0.1, V[b], 3)).max() <= 1e-9
    Gtt, Gt0, G0t, st = dq.greens_tdisplaced_all(_dev(K), 0.1, _dev(V), 3)
    assert int((st != 0).sum()) == 0
    Ott, Ot0 = od.greens_tdisplaced(K, 0.1, V[1], 1)       # every tau
    for l in range(8):
        O0t = od.greens_displaced_back(K, 0.1, V[1], 1, 0, l)
        for got, want in ((Gtt[1, l], Ott[l]), (Gt0[1, l], Ot0[l]), (G0t[1, l], O0t)):
            assert np.abs(got.cpu().numpy() - want).max() <= GTOL * max(1.0, np.abs(want).max())


def test_ended_chains(dq):
    """Groups of a tile whose instance has ended keep their product."""
    N = 150
    K = _hopping(N)
    Vs = [0.3 * di.ising_field(6300 + M, M, N) for M in (3, 4, 8, 17, 5)]
    Gs, ld, sg, st = dq.greens_ragged([(_dev(K), 0.1, _dev(V), 3) for V in Vs])
    assert int((st != 0).sum()) == 0
    for i, V in enumerate(Vs):
        Go, ldo, so = od.greens(K, 0.1, V, 3)
        assert np.abs(Gs[i].cpu().numpy() - Go).max() <= GTOL * max(1.0, np.abs(Go).max())
        assert abs(float(ld[i]) - ldo) <= LTOL * max(1.0, abs(ldo)) and int(sg[i]) == so
