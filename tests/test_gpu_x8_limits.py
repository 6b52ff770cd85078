"""DQMC_CHAIN_BF16X8 at scratch limits, eager and as a graph: a call that fits the
sequential chain's workspace runs there when the tree fold's does not fit."""
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
