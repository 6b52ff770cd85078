"""The QR panel kernel with two CTAs an SM (48 <= N <= 64, launches of many
instances): the same arithmetic as the other form, so an instance's results in a wide
batch are bitwise those in a narrow one, also on the tree fold's row-graded levels."""
import numpy as np
import pytest

import dqmc_inputs as di
from oracle import dqmc as od

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fold,batch", [(0, 300), (1, 75)])
@pytest.mark.parametrize("N", [48, 49, 63, 64])
def test_wide_batch_is_bitwise_narrow(N, fold, batch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2003_05286_gb300 as dq
    K = di.chain_hopping(N)
    V = np.stack([0.5 * di.ising_field(8000 + N + b, 16, N) for b in range(batch)])
    dev = lambda x: torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device="cuda")
    h = dq.Handle(fold=fold)
    G, ld, sg, st = dq.greens(dev(K), 0.1, dev(V), 4, handle=h)
    assert int((st != 0).sum()) == 0
    pick = [0, batch // 2, batch - 1]
    g, l, s, _ = dq.greens(dev(K), 0.1, dev(V[pick]), 4, handle=h)
    assert torch.equal(G[pick], g) and torch.equal(ld[pick], l) and torch.equal(sg[pick], s)
    Go, ldo, so = od.greens(K, 0.1, V[0], 4)
    assert np.abs(G[0].cpu().numpy() - Go).max() <= 1e-10 * max(1.0, np.abs(Go).max())
    assert abs(float(ld[0]) - ldo) <= 1e-9 * max(1.0, abs(ldo)) and int(sg[0]) == so
