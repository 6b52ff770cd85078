"""DQMC_CHAIN_BF16X8 runs on the FP64 chain at every size, tree fold included: the
FP64 tolerances (1e-10 of max(1, max|G|), 1e-9 relative in log det) hold for it."""
import numpy as np
import pytest

import dqmc_inputs as di
from oracle import dqmc as od

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fold", [0, 1])
@pytest.mark.parametrize("N,batch", [(2, 1), (9, 3), (32, 2), (33, 2), (63, 1), (100, 2)])
def test_x8_is_fp64_accurate(N, batch, fold):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2003_05286_gb300 as dq
    K = di.chain_hopping(N)
    V = np.stack([0.3 * di.ising_field(7000 + N + b, 17, N) for b in range(batch)])
    dev = lambda x: torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device="cuda")
    G, ld, sg, st = dq.greens(dev(K), 0.1, dev(V), 4, handle=dq.Handle(chain_precision=8, fold=fold))
    assert int((st != 0).sum()) == 0
    for b in range(batch):
        Go, ldo, so = od.greens(K, 0.1, V[b], 4)
        assert np.abs(G[b].cpu().numpy() - Go).max() <= 1e-10 * max(1.0, np.abs(Go).max())
        assert abs(float(ld[b]) - ldo) <= 1e-9 * max(1.0, abs(ldo)) and int(sg[b]) == so
