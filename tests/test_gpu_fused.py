"""GPU parity of the rows that a sweep combines itself (few pieces a row).

The CTAs of a row block find out which of them is last by counters that belong to the stream and are
0 between calls, whatever ran (or was only captured) on it before: calls of different streams do not
disturb each other, also where one handle names several, and a caller's scratch may hold anything.  The reference is the combining kernel, which a captured call takes and
which has the same bits, or the FP64 oracle.
"""
import math
import threading

import numpy as np
import pytest

from helpers import TOL_D, deff_err

pytestmark = pytest.mark.gpu
K1, K2 = 2 * math.pi / 6.9, 2 * math.pi / 1.55
KAPS = [(K1 * (1 + 0.01 * k), K2) for k in range(4)]


@pytest.fixture(scope="module")
def q():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2511_01255_gb300 as q
    q.lib()
    return q


def pieces(K, NP, N):
    """Pieces of a row at most and whether a CTA's run crosses from one row block into the next."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    smem = lambda W: 1024 + W * 3 * 4096 + 2 * K * 32 * 16 * 24 + W * 3 * 8
    ctas = lambda W: max(1, 232448 // (smem(W) + 1024))
    g = -(-NP // 32)
    few, many = (1, 4) if K == 1 else (2, 8)
    alive = lambda W: W * ctas(W) * g / (-(-g // W) * W)
    W = few if alive(few) > alive(many) else many
    RB, nsub = -(-g // W), -(-N // 32)
    tot, full = RB * nsub, ctas(W) * sms
    C = min(max(1, -(-tot // (full * 60))) * full, max(1, tot // 4))
    start = [tot * x // C for x in range(C + 1)]
    first = {s // nsub for s in start[:-1] if s % nsub == 0}
    q = max(1, tot // C)
    return min(nsub, C, -(-nsub // q) + 1), len(first) < RB


def genes(NP, N, seed):
    import torch
    X = np.random.default_rng(seed).uniform(-1, 1, (NP, N)).astype(np.float32)
    return torch.from_numpy(X).cuda(), X


def captured(call, out):
    """The outputs of one replay of `call`, captured (the combining kernel)."""
    import torch
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        for _ in range(2):  # tables and scratch, then the tables seen complete
            call()
            s.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        call()
    out.fill_(float("nan"))
    g.replay()
    torch.cuda.synchronize()
    return out.clone()


# row blocks that begin inside a CTA's run, with one and with three tables; the last two also have row
# blocks that lie in one run whole
@pytest.mark.parametrize("N,NP,K", [(777, 700, 1), (1100, 5000, 1), (3000, 5000, 3), (590, 3000, 2),
                                    (100, 100000, 1), (90, 70000, 3)])
def test_runs_across_row_blocks_same_bits(q, N, NP, K):
    import torch
    P, crossing = pieces(K, NP, N)
    assert P <= 16 and crossing, (P, crossing)
    X, _ = genes(NP, N, N + K)
    D, f = torch.empty((NP, 2 * K), device="cuda"), torch.empty(NP, device="cuda")

    def call():
        if K == 1:
            q.qpm_eval(N, K1, K2, X, D, f, 1)
        else:
            q.qpm_eval_multi(N, KAPS[:K], X, 1e5, 0.5, f, D)

    ref = captured(call, D)
    for _ in range(3):
        D.fill_(float("nan"))
        call()
        torch.cuda.synchronize()
        assert torch.equal(D, ref)


def multi(q, N, X, K, f, D, scratch, stream=0):
    """qpm_eval_multi through the C entry, with the caller's scratch."""
    probs = (q.Problem * K)(*[(N, a, b) for a, b in KAPS[:K]])
    q._check(q.lib().qpm_eval_multi(probs, K, X.data_ptr(), N, X.shape[0], 1e5, 0.5, D.data_ptr(),
                                    f.data_ptr(), scratch.data_ptr(), scratch.numel(), stream))


@pytest.mark.parametrize("fill", [0, 1, 5, 255])
def test_multi_scratch_holds_anything(q, orc, fill):
    import torch
    K, shapes = 3, [(1000, 300), (129, 129), (640, 900)]
    need = max(q.lib().qpm_eval_multi_scratch_bytes(K, N, NP) for N, NP in shapes)
    scratch = torch.full((need,), fill, dtype=torch.uint8, device="cuda")
    for r in range(2):  # the second round finds the other shapes' sums
        for N, NP in shapes:
            X, Xn = genes(NP, N, N + r)
            D, f = torch.full((NP, K, 2), float("nan"), device="cuda"), torch.empty(NP, device="cuda")
            multi(q, N, X, K, f, D, scratch)
            for k in range(K):
                assert deff_err(D[:, k].cpu().numpy(), orc.deff_closed_genes(Xn, *KAPS[k]), N).max() < TOL_D


def test_multi_on_per_thread_streams(q):
    """The handle of the per-thread default stream names another stream in each thread; with
    scratch of their own the threads' calls are independent."""
    import torch
    K, N, NP, n = 2, 1000, 300, 4
    L = q.lib()
    need = L.qpm_eval_multi_scratch_bytes(K, N, NP)
    work = []
    for t in range(n):
        X, _ = genes(NP, N, t)
        work.append((X, torch.empty(NP, device="cuda"), torch.empty((NP, K, 2), device="cuda"),
                     torch.zeros(need, dtype=torch.uint8, device="cuda")))
    ref = []
    for X, f, D, scratch in work:
        multi(q, N, X, K, f, D, scratch)
        torch.cuda.synchronize()
        ref.append(D.clone())
    bad = []

    def go(t):
        X, f, D, scratch = work[t]
        for _ in range(50):
            D.fill_(float("nan"))
            torch.cuda.synchronize()
            for _ in range(8):
                multi(q, N, X, K, f, D, scratch, 2)  # cudaStreamPerThread
            torch.cuda.synchronize()
            if not torch.equal(D, ref[t]):
                bad.append(t)

    threads = [threading.Thread(target=go, args=(t,)) for t in range(n)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


def test_first_call_of_a_stream_captured(q, orc):
    """A stream whose first call is captured in the relaxed mode, then used eagerly before any
    replay, with memory that has been written before."""
    import torch
    N, NP = 1000, 256
    X, Xn = genes(NP, N, 11)
    D = torch.empty((NP, 2), device="cuda")
    q.qpm_release_caches()
    for _ in range(2):
        q.qpm_eval(N, K1, K2, X, D)  # the tables, on another stream
        torch.cuda.synchronize()
    dirt = [torch.full((1 << 18,), 0x05050505, dtype=torch.int32, device="cuda") for _ in range(8)]
    torch.cuda.synchronize()
    del dirt
    torch.cuda.empty_cache()
    s = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s, capture_error_mode="relaxed"):
        q.qpm_eval(N, K1, K2, X, D)
    ref = orc.deff_closed_genes(Xn, K1, K2)
    for _ in range(2):
        D.fill_(float("nan"))
        torch.cuda.synchronize()
        q.qpm_eval(N, K1, K2, X, D, stream=s)
        torch.cuda.synchronize()
        assert deff_err(D.cpu().numpy(), ref, N).max() < TOL_D
    D.fill_(float("nan"))
    g.replay()
    torch.cuda.synchronize()
    assert deff_err(D.cpu().numpy(), ref, N).max() < TOL_D


def test_more_row_blocks_than_counters(q, orc):
    """Above 4096 row blocks (of 128 rows) the combining kernel takes over."""
    import torch
    N, NP = 40, 4096 * 128 + 6001
    X = torch.empty((NP, N), device="cuda").uniform_(-1, 1, generator=torch.Generator("cuda").manual_seed(2))
    D, f = torch.full((NP, 2), float("nan"), device="cuda"), torch.empty(NP, device="cuda")
    q.qpm_eval(N, K1, K2, X, D, f)
    torch.cuda.synchronize()
    assert not bool(torch.isnan(D).any())
    rows = list(range(0, NP, 5003)) + [4096 * 128 - 1, 4096 * 128, NP - 1]
    ref = orc.deff_closed_genes(X[rows].cpu().numpy(), K1, K2)
    assert deff_err(D[rows].cpu().numpy(), ref, N).max() < TOL_D
