"""Scratch of the tensor-core kernels: what a call's instances need and no more."""
import numpy as np
import pytest

import dqmc_inputs as di

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dq():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2003_05286_gb300 as m
    m.lib()
    return m


def _dev(x):
    return torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device="cuda")


def _fields(seed, batch, M, N):
    return _dev(np.stack([0.3 * di.ising_field(seed + b, M, N) for b in range(batch)]))


def _kernels(fn):
    """Launches of every kernel of one call, by name."""
    from torch.profiler import ProfilerActivity, profile
    for _ in range(2):               # (the first session of a process may come up empty)
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            fn()
            torch.cuda.synchronize()
    out = {e.key: e.count for e in p.key_averages()}
    if not any("dqmc" in k for k in out):
        pytest.skip("no kernel records on this system")
    return out


@pytest.mark.parametrize("N,batch,fold", [(160, 64, 0), (256, 25, 0), (256, 40, 0), (256, 1, 0), (192, 2, 1)])
def test_one_pass_per_solve(dq, N, batch, fold):
    """The two solves of an equal-time call (N >= 160) take all instances in one pass."""
    K, V, h = _dev(di.chain_hopping(N)), _fields(9000, batch, 6, N), dq.Handle(fold=fold)
    runs = _kernels(lambda: dq.greens(K, 0.1, V, 3, handle=h))
    assert sum(n for k, n in runs.items() if "solve_init_kernel" in k) == 2
    assert sum(n for k, n in runs.items() if "lu_kernel" in k) == 0


def test_equal_passes_above_the_cap(dq):
    """N = 384: 512 MB hold 42 solver slots; 85 displaced points and more run in equal
    passes, each point as by itself."""
    N, M = 384, 4
    K, V = _dev(di.chain_hopping(N)), _fields(9100, 20, M, N)
    h = dq.Handle()
    Gtt, Gt0, st = dq.greens_tdisplaced(K, 0.1, V, 1, handle=h)          # 100 points
    assert int((st != 0).sum()) == 0
    for b in (0, 9, 19):
        a, c, _ = dq.greens_tdisplaced(K, 0.1, V[b], 1, handle=dq.Handle())
        assert torch.equal(a, Gtt[b]) and torch.equal(c, Gt0[b])


def test_no_slots_to_spare(dq):
    """One instance of N = 256, sequential fold: 7.1 MB of matrices, 2.1 MB of operand
    digits, 1.1 MB of the slice matrix's, one solver slot of 3.2 MB, and the eighth a
    workspace grows by; a displaced call has QR slots for its instances, not its points."""
    K, V, h = _dev(di.chain_hopping(256)), _fields(9200, 1, 20, 256), dq.Handle(fold=0)
    dq.greens(K, 0.1, V, 5, handle=h)
    assert h.workspace_bytes <= 16 << 20
    # N = 96, 41 points: per point 0.4 MB of digits and 16 matrices; a QR slot is 0.6 MB
    N = 96
    h = dq.Handle()
    dq.greens_tdisplaced(_dev(di.chain_hopping(N)), 0.1, _fields(9300, 1, 40, N), 1, handle=h)
    assert h.workspace_bytes <= 9 / 8 * 41 * (0.4e6 + 22 * 8 * N * N) + (6 << 20)


@pytest.mark.parametrize("jobs,batch", [("2", 9), ("3", 13), ("8", 33), ("8", 39)])
def test_odd_shares(dq, monkeypatch, jobs, batch):
    """Batches that split unevenly into sub-batches: every instance as by itself."""
    N = 160
    K, V = _dev(di.chain_hopping(N)), _fields(9400, batch, 8, N)
    one = [dq.greens(K, 0.1, V[b], 4, handle=dq.Handle(fold=0)) for b in range(batch)]
    monkeypatch.setenv("DQMC_PIPELINE", jobs)
    G, ld, sg, st = dq.greens(K, 0.1, V, 4, handle=dq.Handle(fold=0))
    assert int((st != 0).sum()) == 0
    for b in range(batch):
        assert torch.equal(G[b], one[b][0]) and float(ld[b]) == float(one[b][1])


def test_ragged_groups_share_scratch(dq):
    """24 instances with a K of their own are 24 groups, of which 8 run side by side: those
    past the eighth add their matrices (15 to 18 of N x N), but no digits and no QR slot
    (1.2 MB at N = 96, 16 matrices).  Every instance equals its own call bitwise, also
    among groups of other sizes."""
    N, M = 96, 12
    insts = [(_dev(di.chain_hopping(N)), 0.1, V, 4) for V in _fields(9500, 24, M, N)]
    held = []
    for n in (8, 24):
        h = dq.Handle()
        dq.greens_ragged(insts[:n], handle=h)
        held.append(h.workspace_bytes)
    assert held[1] - held[0] <= 9 / 8 * 16 * 18 * 8 * N * N
    sizes = [40, 64, 64, 96, 130, 160, 200, 64, 256, 33, 96, 48, 160, 20, 64, 300, 72, 100, 64, 161]
    mix = [(_dev(di.chain_hopping(n)), 0.1, _fields(9600 + i, 1, M, n)[0], 4) for i, n in enumerate(sizes)]
    K = _dev(di.chain_hopping(128))
    mix += [(K, 0.1, V, 4) for V in _fields(9700, 11, M, 128)]           # one group, two sub-batches
    for todo in (insts, mix):
        for graphs in (False, True):
            hg = dq.Handle(graphs=graphs)
            for _ in range(2):
                G, ld, sg, st = dq.greens_ragged(todo, handle=hg)
            assert int((st != 0).sum()) == 0
            for i, (K1, dt, V1, k) in enumerate(todo):
                G1, ld1, _, _ = dq.greens(K1, dt, V1, k, handle=dq.Handle(fold=0))
                assert torch.equal(G1, G[i]) and float(ld1) == float(ld[i])


@pytest.mark.parametrize("graphs", [False, True])
def test_full_device_keeps_the_workspace(dq, graphs):
    """128 instances of N = 256 on a device with 300 MB too little for the whole workspace
    (0.7 GB of digits beside 0.9 GB of matrices).  The calls run without the digits, and after the first one none of them
    allocates or frees device memory."""
    from torch.profiler import ProfilerActivity, profile
    N, M, batch = 256, 4, 128
    K, V = _dev(di.chain_hopping(N)), _fields(9800, batch, M, N)
    h0 = dq.Handle(fold=0)
    ref = dq.logdet(K, 0.1, V, 2, handle=h0)
    full = h0.workspace_bytes
    h0.close()
    h = dq.Handle(fold=0, graphs=graphs)
    dq.logdet(K, 0.1, V[:1], 2, handle=h)          # loads the kernels
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    room = full * 8 // 9 - (300 << 20)             # too little for the digits by 300 MB
    fill = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
    try:
        ld, sg, st = dq.logdet(K, 0.1, V, 2, handle=h)
        held = h.workspace_bytes
        assert held < room and int((st != 0).sum()) == 0
        for _ in range(2):
            with profile(activities=[ProfilerActivity.CPU, ProfilerActivity.CUDA]) as p:
                ld, sg, st = dq.logdet(K, 0.1, V, 2, handle=h)
                torch.cuda.synchronize()
        names = {e.key for e in p.key_averages()}
        assert any("cuda" in n for n in names)
        assert not names & {"cudaFree", "cudaMalloc"}
        assert h.workspace_bytes == held
        assert ((ld - ref[0]).abs() <= 1e-9 * ref[0].abs()).all() and torch.equal(sg, ref[1])
    finally:
        del fill
        torch.cuda.empty_cache()


@pytest.mark.parametrize("prec", [0, 8])
@pytest.mark.parametrize("call", ["greens", "displaced", "gradient"])
@pytest.mark.parametrize("N", [64, 160])
def test_no_room_means_the_fp64_pipe(dq, N, call, prec):
    """Under a limit that leaves no room for the digits no tensor-core kernel runs, and
    without the limit they do: the fallback is what ran."""
    K, V = _dev(di.chain_hopping(N)), _fields(9900 + N, 3, 8, N)
    run = {"greens": dq.greens, "displaced": dq.greens_tdisplaced, "gradient": dq.logdet_grad}[call]
    names = ("tc_gemm_kernel", "chain_tc_kernel", "qr_panel_kernel", "qr_apply_kernel", "solve_back_kernel")
    free = dq.Handle(fold=0, chain_precision=prec)
    ref = run(K, 0.1, V, 4, handle=free)
    with_room = _kernels(lambda: run(K, 0.1, V, 4, handle=free))
    assert any(n in k for k in with_room for n in names)
    h = dq.Handle(fold=0, chain_precision=prec)
    # one digit operand of one instance (8 planes of N padded to 128 by 32) too little
    h.set_memory_limit(free.device_bytes * 8 // 9 - 16 * ((N + 127) // 128 * 128) * ((N + 31) // 32 * 32))
    without = _kernels(lambda: run(K, 0.1, V, 4, handle=h))
    assert not any(n in k for k in without for n in names)
    out = run(K, 0.1, V, 4, handle=h)
    assert (out[0] - ref[0]).abs().max().item() <= 1e-9 * max(1.0, ref[0].abs().max().item())
