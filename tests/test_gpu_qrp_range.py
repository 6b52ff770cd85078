"""Scales near both ends of FP64's range in the factorisations and solves: chunk products
of norm e^{+-340} and e^{+-348}, whose squares (1e295 to 1e303 and their inverses) a
reflector may not rely on.  Closed forms of the non-interacting problem, site by
site uniform or with two decoupled sublattices of opposite fields; the suite's tolerances
(1e-10 in G, 1e-9 relative in log det)."""
import numpy as np
import pytest

import dqmc_inputs as di
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


# fields of one slice, ten slices a chunk, in units of the amplitude
PATTERNS = {"up": [1], "down up": [-1, 1], "up down": [1, -1], "rise fall": [.5, .5, -.5, -.5],
            "four": [-1, 1, -1, 1]}


@pytest.mark.parametrize("fold", [0, 1])
@pytest.mark.parametrize("amp", [34.0, 34.8])
@pytest.mark.parametrize("pattern", list(PATTERNS))
@pytest.mark.parametrize("N", [48, 64, 100, 160, 257, 384])
def test_uniform_fields(dq, N, pattern, amp, fold):
    K = di.chain_hopping(N)
    c = amp * np.repeat(PATTERNS[pattern], 10)
    V = np.repeat(c[:, None], N, axis=1)
    G, ld, sg, st = dq.greens(_dev(K), 0.1, _dev(V), 10, handle=dq.Handle(fold=fold))
    Gx, ldx = ex.closed_form_greens(K, 0.1 * len(c), shift=c.sum())
    assert int(st) == 0
    assert np.abs(G.cpu().numpy() - Gx).max() <= GTOL
    assert abs(float(ld) - ldx) <= LTOL * max(1.0, abs(ldx)) and int(sg) == 1


def _sublattices(N):
    """Two rings of N / 2 sites, one on the even sites, one on the odd ones."""
    K = np.zeros((N, N))
    K[0::2, 0::2] = K[1::2, 1::2] = di.chain_hopping(N // 2)
    return K


@pytest.mark.parametrize("fold", [0, 1])
@pytest.mark.parametrize("N", [64, 80, 130, 200])
def test_opposite_fields(dq, N, fold):
    """Columns of norm e^{348} and e^{-348} in one factorisation (N > 64: in one panel)."""
    K, a = _sublattices(N), 34.8
    s = np.where(np.arange(N) % 2 == 0, 1.0, -1.0)
    V = np.repeat([a, 0.0], 10)[:, None] * s[None]
    G, ld, sg, st = dq.greens(_dev(K), 0.1, _dev(V), 10, handle=dq.Handle(fold=fold))
    assert int(st) == 0
    G, ldx = G.cpu().numpy(), 0.0
    for o, shift in ((0, 10 * a), (1, -10 * a)):
        Gx, l = ex.closed_form_greens(di.chain_hopping(N // 2), 2.0, shift=shift)
        assert np.abs(G[o::2, o::2] - Gx).max() <= GTOL and np.abs(G[o::2, 1 - o::2]).max() <= GTOL
        ldx += l
    assert abs(float(ld) - ldx) <= LTOL * abs(ldx) and int(sg) == 1


@pytest.mark.parametrize("N", [64, 160, 192])
def test_displaced_and_gradient(dq, N):
    """Both stacks and the two-stack solves at these scales (N >= 160: the QR solver)."""
    K = di.chain_hopping(N)
    c = np.repeat([34.8, -34.8], 10)
    V = np.repeat(c[:, None], N, axis=1)
    Gtt, Gt0, st = dq.greens_tdisplaced(_dev(K), 0.1, _dev(V), 10)
    assert int(st) == 0
    Gx, ldx = ex.closed_form_greens(K, 2.0)
    for j in range(Gtt.shape[0]):
        assert np.abs(Gtt[j].cpu().numpy() - Gx).max() <= GTOL
        tau = 10 * j
        want = ex.closed_form_displaced(K, 2.0, 0.1 * tau, 0.0, c[:tau].sum())
        assert np.abs(Gt0[j].cpu().numpy() - want).max() <= GTOL * max(1.0, np.abs(want).max())
    ld, sg, dV, st = dq.logdet_grad(_dev(K), 0.1, _dev(V), 10)
    assert int(st) == 0 and abs(float(ld) - ldx) <= LTOL * abs(ldx) and int(sg) == 1
    # d log det / d V_l(i) = 1 - G_ii, the same at every slice
    assert np.abs(dV.cpu().numpy() - (1.0 - np.diag(Gx))[None]).max() <= 1e-9
