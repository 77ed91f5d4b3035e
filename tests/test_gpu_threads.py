"""Host threads with a stream each: every call's results are those of the call alone."""
import math
import threading
from types import SimpleNamespace

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
K1, K2 = 2 * math.pi / 6.9, 2 * math.pi / 1.55


@pytest.fixture(scope="module")
def q():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2511_01255_gb300 as q
    q.lib()
    return q


@pytest.mark.parametrize("kind", ["eval", "packed"])
@pytest.mark.parametrize("N,NP", [(20000, 600), (1000, 300)])
def test_per_thread_default_streams(q, kind, N, NP):
    """cudaStreamPerThread is one handle for all threads and another stream in each."""
    import torch
    mine, n = SimpleNamespace(cuda_stream=2), 4
    rng = np.random.default_rng(N)
    work = []
    for t in range(n):
        if kind == "eval":
            X = torch.from_numpy(rng.uniform(-1, 1, (NP, N)).astype(np.float32)).cuda()
        else:
            X = torch.from_numpy(rng.integers(-2**31, 2**31, (NP, (N + 31) // 32)).astype(np.int32)).cuda()
        D = torch.empty((NP, 2), device="cuda")
        call = q.qpm_eval if kind == "eval" else q.qpm_eval_packed
        call(N, K1, K2, X, D)
        torch.cuda.synchronize()
        work.append((call, X, D, D.clone()))
    bad = []

    def go(t):
        call, X, D, ref = work[t]
        for _ in range(30):
            D.fill_(float("nan"))
            torch.cuda.synchronize()
            for _ in range(8):
                call(N, K1, K2, X, D, stream=mine)
            torch.cuda.synchronize()
            if not torch.equal(D, ref):
                bad.append(t)

    threads = [threading.Thread(target=go, args=(t,)) for t in range(n)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


def test_many_threads_one_after_the_other(q):
    """More threads than scratch buffers are kept for."""
    import torch
    N, NP, mine = 2000, 300, SimpleNamespace(cuda_stream=2)
    X = torch.from_numpy(np.random.default_rng(1).uniform(-1, 1, (NP, N)).astype(np.float32)).cuda()
    ref, D = torch.empty((NP, 2), device="cuda"), torch.empty((NP, 2), device="cuda")
    q.qpm_eval(N, K1, K2, X, ref)
    torch.cuda.synchronize()
    for _ in range(80):
        D.fill_(float("nan"))
        torch.cuda.synchronize()
        t = threading.Thread(target=lambda: q.qpm_eval(N, K1, K2, X, D, stream=mine))
        t.start()
        t.join()
        torch.cuda.synchronize()
        assert torch.equal(D, ref)


@pytest.mark.parametrize("ld", [512, 513])
@pytest.mark.parametrize("kind", ["eval", "packed", "multi", "shg", "relaxed"])
def test_first_cuda_call_of_a_thread(q, kind, ld):
    """A thread whose first CUDA call is one of the library's, with every table and buffer there."""
    import torch
    N, NP = 512, 200
    X = torch.from_numpy(np.random.default_rng(ld).uniform(-1, 1, (NP, ld)).astype(np.float32)).cuda()[:, :N]
    words = torch.arange(NP * 16, dtype=torch.int32, device="cuda").view(NP, 16)
    D, f, M = (torch.empty(s, device="cuda") for s in ((NP, 2), (NP,), (NP, 2, 2)))
    S, g, one = q.relaxed_saved(NP, N), torch.empty((NP, ld), device="cuda")[:, :N], torch.ones(NP, device="cuda")
    L, kaps = q.lib(), (q.Problem * 2)((N, K1, K2), (N, K1 * 1.01, K2))
    need = L.qpm_eval_multi_scratch_bytes(2, N, NP)
    scratch = torch.empty(need, dtype=torch.uint8, device="cuda")
    ptr = [t.data_ptr() for t in (X, words, D, f, M, S, g, one, scratch)]
    x, w, d, fp, m, s, gp, o, sc = ptr
    calls = {  # through the C entries: the tensors' own checks make CUDA calls
        "eval": lambda: L.qpm_eval(kaps, x, ld, NP, d, fp, 0, None),
        "packed": lambda: L.qpm_eval_packed(kaps, w, 16, NP, d, fp, 0, None),
        "multi": lambda: L.qpm_eval_multi(kaps, 2, x, ld, NP, 1e4, 0.5, m, fp, sc, need, None),
        "shg": lambda: L.qpm_eval_shg(kaps, x, ld, NP, d, fp, None),
        "relaxed": lambda: (L.qpm_deff_relaxed_fwd(kaps, x, ld, NP, d, fp, s, None) or
                            L.qpm_deff_relaxed_bwd(kaps, x, ld, NP, d, s, o, gp, ld, None))}
    outs = {"multi": [M, f], "relaxed": [D, f, g]}.get(kind, [D, f])
    for _ in range(2):
        assert calls[kind]() == 0
        torch.cuda.synchronize()
    ref, got = [t.clone() for t in outs], []
    for t in outs:
        t.fill_(float("nan"))
    torch.cuda.synchronize()
    t = threading.Thread(target=lambda: got.append((calls[kind](), L.qpm_last_error())))
    t.start()
    t.join()
    torch.cuda.synchronize()
    assert got[0][0] == 0, got
    for a, b in zip(outs, ref):
        assert torch.equal(a, b)


@pytest.mark.parametrize("plain", [False, True])
def test_multi_scratch_lives_until_its_stream_is_done(q, plain):
    """qpm_eval_multi's scratch comes from the current stream's pool and is used on `stream`: memory
    of the same size taken on the current stream meanwhile is other memory."""
    import torch
    N, NP, K = 100000, 512, 2
    kaps = [(K1, K2), (K1 * 1.01, K2)]
    X = torch.empty((NP, N), device="cuda").uniform_(-1, 1, generator=torch.Generator("cuda").manual_seed(3))
    D, f = torch.empty((NP, K, 2), device="cuda"), torch.empty(NP, device="cuda")
    q.qpm_eval_multi(N, kaps, X, 1e5, 0.5, f, D)
    torch.cuda.synchronize()
    ref, need = D.clone(), q.lib().qpm_eval_multi_scratch_bytes(K, N, NP)
    side = torch.cuda.Stream()
    s = SimpleNamespace(cuda_stream=side.cuda_stream) if plain else side  # any object with the handle
    for _ in range(20):
        torch.cuda.synchronize()
        for _ in range(4):
            q.qpm_eval_multi(N, kaps, X, 1e5, 0.5, f, D, stream=s)
        for _ in range(30):
            torch.empty(need, dtype=torch.uint8, device="cuda").fill_(255)
        torch.cuda.synchronize()
        assert torch.equal(D, ref)


@pytest.mark.parametrize("N,NP", [(30000, 300), (2000, 300)])
def test_destroyed_streams_whose_handle_comes_back(q, N, NP):
    """A stream is destroyed with its calls still pending; the next stream often has its handle."""
    import ctypes
    import torch
    rt = torch.cuda.cudart()
    rng = np.random.default_rng(N)
    X = [torch.from_numpy(rng.uniform(-1, 1, (NP, N)).astype(np.float32)).cuda() for _ in range(2)]
    ref = [torch.empty((NP, 2), device="cuda") for _ in range(2)]
    for x, r in zip(X, ref):
        q.qpm_eval(N, K1, K2, x, r)
    D = [torch.empty((NP, 2), device="cuda") for _ in range(2)]
    handles = set()
    for _ in range(100):  # more streams than scratch buffers of ended ones are kept
        for d in D:
            d.fill_(float("nan"))
        torch.cuda.synchronize()
        for x, d in zip(X, D):
            h = ctypes.c_void_p()
            assert int(rt.cudaStreamCreate(ctypes.addressof(h))) == 0
            handles.add(h.value)
            for _ in range(5):
                q.qpm_eval(N, K1, K2, x, d, stream=SimpleNamespace(cuda_stream=h.value))
            assert int(rt.cudaStreamDestroy(h.value)) == 0
        torch.cuda.synchronize()
        for d, r in zip(D, ref):
            assert torch.equal(d, r)
    assert len(handles) < 200  # some came back
