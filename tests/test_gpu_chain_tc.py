"""The fused chunk chain on the tensor cores (33 <= N <= 128): one to four 32-row
K-blocks with remainders, one to four column blocks, chunks of one slice, of many and
ragged ones, both directions, the tree fold, ended chains, non-finite fields.

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


def _hopping(N):
    return di.chain_hopping(N) + np.diag(0.2 * np.cos(np.arange(N)))


def _check(G, ld, sg, K, V, k):
    Go, ldo, so = od.greens(K, 0.1, V, k)
    assert np.abs(G - Go).max() <= GTOL * max(1.0, np.abs(Go).max())
    assert abs(ld - ldo) <= LTOL * max(1.0, abs(ldo)) and sg == so


@pytest.mark.parametrize("fold", [0, 1])
@pytest.mark.parametrize("N,M,k", [(33, 9, 4), (36, 3, 1), (63, 12, 12), (64, 11, 5), (65, 7, 3),
                                   (96, 4, 1), (97, 10, 5), (101, 9, 4), (127, 6, 3), (128, 13, 10)])
def test_greens(dq, N, M, k, fold):
    K = _hopping(N)
    V = np.stack([0.3 * di.ising_field(5000 + N + b, M, N) for b in range(3)])
    G, ld, sg, st = dq.greens(_dev(K), 0.1, _dev(V), k, handle=dq.Handle(fold=fold))
    assert int((st != 0).sum()) == 0
    for b in range(3):
        _check(G[b].cpu().numpy(), float(ld[b]), int(sg[b]), K, V[b], k)


@pytest.mark.parametrize("N", [40, 64, 100])
def test_both_directions(dq, N):
    K, V = _hopping(N), 0.3 * di.ising_field(5200 + N, 11, N)
    Gtt, Gt0, G0t, st = dq.greens_tdisplaced(_dev(K), 0.1, _dev(V), 4, want_0t=True)
    assert int(st) == 0
    Ott, Ot0 = od.greens_tdisplaced(K, 0.1, V, 4)
    for j, l in enumerate(od.tau_grid(11, 4)):
        O0t = od.greens_displaced_back(K, 0.1, V, 4, 0, l)
        for got, want in ((Gtt[j], Ott[j]), (Gt0[j], Ot0[j]), (G0t[j], O0t)):
            assert np.abs(got.cpu().numpy() - want).max() <= GTOL * max(1.0, np.abs(want).max())


@pytest.mark.parametrize("N", [45, 128])
def test_ended_chains(dq, N):
    """Instances of one group with different M: some end in front of a chunk, some inside."""
    K = _hopping(N)
    Vs = [0.3 * di.ising_field(5300 + M, M, N) for M in (3, 4, 8, 17)]
    Gs, ld, sg, st = dq.greens_ragged([(_dev(K), 0.1, _dev(V), 3) for V in Vs])
    assert int((st != 0).sum()) == 0
    for i, V in enumerate(Vs):
        _check(Gs[i].cpu().numpy(), float(ld[i]), int(sg[i]), K, V, 3)


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_non_finite_field(dq, value):
    """A non-finite entry is flagged for its instance and leaves the other one alone."""
    N, K = 48, _hopping(48)
    V = np.stack([0.3 * di.ising_field(5400 + b, 8, N) for b in range(2)])
    V[1, 3, 7] = value
    G, ld, sg, st = dq.greens(_dev(K), 0.1, _dev(V), 4, handle=dq.Handle(fold=0))
    assert int(st[0]) == 0 and int(st[1]) != 0
    _check(G[0].cpu().numpy(), float(ld[0]), int(sg[0]), K, V[0], 4)
    assert not bool(torch.isfinite(G[1]).all())
