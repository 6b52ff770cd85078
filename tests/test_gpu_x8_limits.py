"""DQMC_CHAIN_BF16X8 at scratch limits, eager and as a graph: a call that fits the
sequential chain's workspace runs there when the tree fold's does not fit, and at every
limit the graph runs the same kernels as the eager call."""
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


@pytest.mark.parametrize("fold", [1, 2])
@pytest.mark.parametrize("N,graphs", [(16, False), (16, True), (48, False), (96, False)])
def test_sequential_where_the_tree_does_not_fit(dq, N, graphs, fold):
    """The sequential chain takes below 24 N x N matrices, the tree of 12 chunks over 100."""
    K, V = di.chain_hopping(N), 0.3 * di.ising_field(8000 + N, 60, N)
    Go, ldo, so = od.greens(K, 0.1, V, 5)
    h = dq.Handle(chain_precision=8, graphs=graphs, fold=fold)
    h.set_memory_limit(24 * 8 * N * N + 2 * 8 * 60 * N + 64 * 256)
    for _ in range(2):
        G, ld, sg, st = dq.greens(_dev(K), 0.1, _dev(V), 5, handle=h)
        assert int(st) == 0 and int(sg) == so
        assert np.abs(G.cpu().numpy() - Go).max() <= GTOL * max(1.0, np.abs(Go).max())
        assert abs(float(ld) - ldo) <= LTOL * max(1.0, abs(ldo))
    # an FP64 call whose tree does not fit stays refused
    h = dq.Handle(graphs=graphs, fold=2)
    h.set_memory_limit(24 * 8 * N * N + 2 * 8 * 60 * N + 64 * 256)
    with pytest.raises(RuntimeError, match="allocation failed"):
        dq.greens(_dev(K), 0.1, _dev(V), 5, handle=h)


@pytest.mark.parametrize("prec", [0, 8])
@pytest.mark.parametrize("N,batch,M", [(48, 1, 60), (64, 3, 40), (64, 32, 40), (100, 2, 40), (160, 1, 40)])
def test_graph_is_the_eager_call_at_every_limit(dq, N, batch, M, prec):
    """Limits between the smallest and the whole workspace: the graph succeeds where the
    eager call does, with the same bits, also where there is no room for the digits."""
    K = _dev(di.chain_hopping(N))
    V = _dev(np.stack([0.3 * di.ising_field(8100 + N + b, M, N) for b in range(batch)]))
    free = dq.Handle(chain_precision=prec)
    ref = dq.greens(K, 0.1, V, 5, handle=free)
    done = 0
    for share in (1.0, 0.7, 0.5, 0.35, 0.25, 0.18, 0.12, 0.08, 0.05):
        out = []
        for graphs in (False, True):
            h = dq.Handle(chain_precision=prec, graphs=graphs)
            h.set_memory_limit(int(free.device_bytes * share))
            try:
                G, ld, sg, st = dq.greens(K, 0.1, V, 5, handle=h)
            except RuntimeError as e:
                assert "allocation failed" in str(e)
                out.append(None)
                continue
            assert int((st != 0).sum()) == 0
            assert (G - ref[0]).abs().max().item() <= GTOL * max(1.0, ref[0].abs().max().item())
            out.append((G, ld, sg))
        assert (out[0] is None) == (out[1] is None)
        if out[0] is not None:
            assert all(torch.equal(a, b) for a, b in zip(*out))
            done += 1
    assert done >= 3


@pytest.mark.parametrize("N", [36, 48, 96])
def test_graph_without_digits_is_fp64_accurate(dq, N):
    """The smallest workspace of all, as a graph."""
    K, V = di.chain_hopping(N), 0.3 * di.ising_field(8200 + N, 60, N)
    Go, ldo, so = od.greens(K, 0.1, V, 5)
    h = dq.Handle(chain_precision=8, graphs=True)
    h.set_memory_limit(24 * 8 * N * N + 2 * 8 * 60 * N + 64 * 256)
    for _ in range(2):
        G, ld, sg, st = dq.greens(_dev(K), 0.1, _dev(V), 5, handle=h)
        assert int(st) == 0 and int(sg) == so
        assert np.abs(G.cpu().numpy() - Go).max() <= GTOL * max(1.0, np.abs(Go).max())
        assert abs(float(ld) - ldo) <= LTOL * max(1.0, abs(ldo))
