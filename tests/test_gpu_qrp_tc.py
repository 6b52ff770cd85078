"""Blocked pivoted QR on the tensor cores (64 <= N <= 384), through the calls that
use it: edges of its 32-column panels and 128-row tiles and of its N range, both
folds (the tree's levels have row-graded matrices), scales up to e^{+-200},
columns that vanish, and more instances than one pass of its workspace holds.

The tolerances are the suite's, 1e-10 of max(1, max|G|) and 1e-9 relative in log
det, against the FP64 oracle or a closed form."""
import numpy as np
import pytest

import dqmc_inputs as di
from oracle import dqmc as od
from oracle import exact as ex

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


@pytest.mark.parametrize("fold", [0, 1])
@pytest.mark.parametrize("N", [64, 65, 95, 97, 128, 160, 161, 192, 193, 224, 256, 257, 320, 384, 385])
def test_panel_edges(dq, N, fold):
    """Four chunks of strongly graded fields: pivoting mixes the panels."""
    K = di.chain_hopping(N)
    V = np.stack([0.5 * di.ising_field(5000 + N + b, 20, N) for b in range(2)])
    G, ld, sg, st = dq.greens(_dev(K), 0.2, _dev(V), 5, handle=dq.Handle(fold=fold))
    assert int((st != 0).sum()) == 0
    for b in range(2):
        Go, ldo, so = od.greens(K, 0.2, V[b], 5)
        assert np.abs(G[b].cpu().numpy() - Go).max() <= GTOL * max(1.0, np.abs(Go).max())
        assert abs(float(ld[b]) - ldo) <= LTOL * abs(ldo) and int(sg[b]) == so


@pytest.mark.parametrize("fold", [0, 1])
@pytest.mark.parametrize("L", [8, 12])
def test_closed_form_beta50(dq, L, fold):
    """U = 0 with a site-independent field at beta = 50 (scales e^{+-200})."""
    K = di.square_hopping(L)
    N, M = L * L, 500
    c = np.random.default_rng(L).uniform(-0.3, 0.3, M)
    V = np.repeat(c[:, None], N, axis=1)
    G, ld, sg, st = dq.greens(_dev(K), 0.1, _dev(V), 10, handle=dq.Handle(fold=fold))
    Gx, ldx = ex.closed_form_greens(K, 50.0, shift=c.sum())
    assert int(st) == 0
    assert np.abs(G.cpu().numpy() - Gx).max() <= GTOL
    assert abs(float(ld) - ldx) <= LTOL * max(1.0, abs(ldx))


@pytest.mark.parametrize("fold", [0, 1])
def test_vanishing_column(dq, fold):
    """e^V = 0 at one site of one instance: flagged there, the other instance untouched."""
    N = 96
    K = di.chain_hopping(N)
    V = np.stack([0.3 * di.ising_field(5100 + b, 16, N) for b in range(2)])
    bad = V.copy()
    bad[1, :, 5] = -1e4
    G, ld, sg, st = dq.greens(_dev(K), 0.1, _dev(bad), 4, handle=dq.Handle(fold=fold))
    assert int(st[0]) == 0 and int(st[1]) != 0
    Go, ldo, so = od.greens(K, 0.1, V[0], 4)
    assert np.abs(G[0].cpu().numpy() - Go).max() <= GTOL
    assert abs(float(ld[0]) - ldo) <= LTOL * abs(ldo) and int(sg[0]) == so


def test_more_instances_than_slots(dq):
    """N = 384: the workspace holds fewer slots than there are instances; every
    instance equals its own call bitwise."""
    N = 384
    K = _dev(di.chain_hopping(N))
    V = _dev(np.stack([0.3 * di.ising_field(5200 + b, 6, N) for b in range(130)]))
    h = dq.Handle(fold=0)
    G, ld, sg, st = dq.greens(K, 0.1, V, 3, handle=h)
    assert int((st != 0).sum()) == 0
    for b in (0, 64, 129):
        G1, ld1, _, _ = dq.greens(K, 0.1, V[b], 3, handle=dq.Handle(fold=0))
        assert torch.equal(G1, G[b]) and float(ld1) == float(ld[b])


@pytest.mark.parametrize("N", [160, 161, 257])
def test_solver_through_displaced_and_gradient(dq, N):
    """The QR solver (N >= 160) with 2 N right-hand sides, and with none (log det alone)."""
    K = di.chain_hopping(N)
    V = 0.3 * di.ising_field(5300 + N, 7, N)
    Gtt, Gt0, st = dq.greens_tdisplaced(_dev(K), 0.1, _dev(V), 3)
    assert int(st) == 0
    Ott, Ot0 = od.greens_tdisplaced(K, 0.1, V, 3)
    for got, want in ((Gtt, Ott), (Gt0, Ot0)):
        assert np.abs(got.cpu().numpy() - want).max() <= GTOL * max(1.0, np.abs(want).max())
    ldo, so = od.logdet(K, 0.1, V, 3)
    ld, sg, st = dq.logdet(_dev(K), 0.1, _dev(V), 3)
    assert int(st) == 0 and abs(float(ld) - ldo) <= LTOL * abs(ldo) and int(sg) == so
    ld, sg, dV, st = dq.logdet_grad(_dev(K), 0.1, _dev(V), 3)
    assert int(st) == 0 and abs(float(ld) - ldo) <= LTOL * abs(ldo) and int(sg) == so
    assert np.abs(dV.cpu().numpy() - od.logdet_grad(K, 0.1, V, 3)).max() <= 1e-9


def test_solver_sign(dq):
    """Negative determinants at N = 160: the sign comes from the reflectors and R."""
    N = 160
    K = np.zeros((N, N))
    K[:3, :3] = di.chain_hopping(3)          # a triangle with strong fields, the rest decoupled
    signs = set()
    for seed in range(24):
        V = np.zeros((6, N))
        V[:, :3] = 2.0 * di.gaussian_field(seed, 6, 3)
        ld, sg, st = dq.logdet(_dev(K), 0.5, _dev(V), 2)
        ldo, so = od.logdet(K, 0.5, V, 2)
        assert int(st) == 0 and int(sg) == so and abs(float(ld) - ldo) <= LTOL * abs(ldo)
        signs.add(int(sg))
    assert signs == {-1, 1}
