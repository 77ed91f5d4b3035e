"""Captured calls: what a graph was given stays its own for as long as it exists.

A call made on a capturing stream leaves addresses of tables and scratch in the graph.  They have
to stay valid past calls that replace the stream's scratch, past eviction and qpm_release_caches,
and replays may run beside other calls of the captured stream; with the graph they are given back.
The reference is the same call made eagerly (the same bits) or the FP64 oracle.
"""
import math
import time

import numpy as np
import pytest

from helpers import TOL_D, deff_err

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


def genes(NP, N, seed=0):
    import torch
    X = np.random.default_rng(seed).uniform(-1, 1, (NP, N)).astype(np.float32)
    return torch.from_numpy(X).cuda(), X


def calls(q, N, NP):
    """name -> (call, outputs) of every entry point that may be captured."""
    import torch
    X, _ = genes(NP, N, N)
    words = torch.randint(-2**31, 2**31 - 1, (NP, (N + 31) // 32), dtype=torch.int32, device="cuda")
    new = lambda *s: torch.empty(s, device="cuda")
    D, f, P, M, fm, E = new(NP, 2), new(NP), new(NP, 2), new(NP, 3, 2), new(NP), new(NP, 2)
    S, R, g, one = q.relaxed_saved(NP, N), new(NP, 2), new(NP, N), torch.ones(NP, device="cuda")
    kaps = [(K1 + 0.01 * k, K2) for k in range(3)]

    def pair():
        q.qpm_deff_relaxed_fwd(N, K1, K2, X, R, None, S)
        q.qpm_deff_relaxed_bwd(N, K1, K2, X, R, S, one, g)

    return {"eval": (lambda: q.qpm_eval(N, K1, K2, X, D, f, 1), [D, f]),
            "packed": (lambda: q.qpm_eval_packed(N, K1, K2, words, P), [P]),
            "multi": (lambda: q.qpm_eval_multi(N, kaps, X, 1e5, 0.5, fm, M), [fm, M]),
            "shg": (lambda: q.qpm_eval_shg(N, K1, X, E), [E]),
            "relaxed": (pair, [R, g])}


def capture(call, stream, **kw):
    import torch
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream, **kw):
        call()
    return g


NAMES = ["eval", "packed", "multi", "shg", "relaxed"]


@pytest.mark.parametrize("mode", ["global", "relaxed"])
@pytest.mark.parametrize("name", NAMES)
def test_graph_outlives_the_caches(q, name, mode):
    import torch
    call, outs = calls(q, 2000, 300)[name]
    q.qpm_release_caches()
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    g = capture(call, s, capture_error_mode=mode)  # the first call: no tables, no scratch
    call()  # finds the tables the capture built
    torch.cuda.synchronize()
    ref = [o.clone() for o in outs]
    with torch.cuda.stream(s):  # this stream's scratch comes and grows
        for NP in (64, 4000):
            X, _ = genes(NP, 1500)
            q.qpm_eval(1500, K1, K2, X, torch.empty((NP, 2), device="cuda"), None, 1)
    s.synchronize()
    X, _ = genes(4, 40)
    for k in range(70):  # more problems than the cache holds
        q.qpm_eval(40, K1 + 0.001 * k, K2, X, torch.empty((4, 2), device="cuda"))
    q.qpm_release_caches()
    dirt = [torch.full((n,), float("nan"), device="cuda") for n in (1 << 8, 1 << 12, 1 << 16, 1 << 19) * 12]
    for _ in range(2):
        for o in outs:
            o.fill_(float("nan"))
        g.replay()
        torch.cuda.synchronize()
        for o, r in zip(outs, ref):
            assert torch.equal(o, r)
    assert all(bool(torch.isnan(d).all()) for d in dirt)
    call()
    torch.cuda.synchronize()
    for o, r in zip(outs, ref):
        assert torch.equal(o, r)


@pytest.mark.parametrize("name", ["eval", "packed"])
def test_replays_beside_calls_of_the_captured_stream(q, name):
    import torch
    a, b = calls(q, 3000, 1500), calls(q, 2500, 1400)
    (call, outs), (other, outs2) = a[name], b[name]
    call(), other()
    torch.cuda.synchronize()
    ref, ref2 = [o.clone() for o in outs], [o.clone() for o in outs2]
    s, r = torch.cuda.Stream(), torch.cuda.Stream()
    g = capture(lambda: (call(), call()), s)  # two calls of one stream share the graph's scratch
    for _ in range(20):
        for o in outs + outs2:
            o.fill_(float("nan"))
        torch.cuda.synchronize()
        with torch.cuda.stream(r):
            for _ in range(4):
                g.replay()
        with torch.cuda.stream(s):
            for _ in range(8):
                other()
        torch.cuda.synchronize()
        for o, x in zip(outs + outs2, ref + ref2):
            assert torch.equal(o, x)


def test_two_captured_streams_of_one_graph(q):
    """Parallel branches of a capture, each on a stream of its own."""
    import torch
    (c1, o1), (c2, o2) = calls(q, 3000, 900)["eval"], calls(q, 2500, 1100)["eval"]
    c1(), c2()
    torch.cuda.synchronize()
    ref = [o.clone() for o in o1 + o2]
    s, t = torch.cuda.Stream(), torch.cuda.Stream()

    def fork():
        t.wait_stream(s)
        c1()
        with torch.cuda.stream(t):
            c2()
        s.wait_stream(t)

    g = capture(fork, s)
    for _ in range(10):
        for o in o1 + o2:
            o.fill_(float("nan"))
        g.replay()
        torch.cuda.synchronize()
        for o, x in zip(o1 + o2, ref):
            assert torch.equal(o, x)


@pytest.mark.parametrize("n", [1, 70])
def test_full_cache(q, orc, n):
    """Problems that no longer fit the cache, first met in a capture: the first 64 of them still go
    there, the others' tables are the graph's alone.  Each is used twice."""
    import torch
    q.qpm_release_caches()
    X, Xn = genes(40, 300)
    D, E = torch.empty((40, 2), device="cuda"), torch.empty((n, 40, 2), device="cuda")
    for k in range(64):
        q.qpm_eval(300, K1 + 0.001 * k, K2, X, D)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()

    def call():
        for k in range(n):
            q.qpm_eval(300, K1 / 2 + 0.001 * k, K2, X, D)
            q.qpm_eval(300, K1 / 2 + 0.001 * k, K2, X, E[k])

    g = capture(call, s)
    for _ in range(2):
        E.fill_(float("nan"))
        g.replay()
        torch.cuda.synchronize()
        for k in (0, n // 2, n - 1):
            ref = orc.deff_closed_genes(Xn, K1 / 2 + 0.001 * k, K2)
            assert deff_err(E[k].cpu().numpy(), ref, 300).max() < TOL_D
        q.qpm_eval(300, K1 / 3, K2, X, D)  # evicts what no graph holds
        q.qpm_release_caches()


def test_memory_comes_back_with_the_graph(q):
    """The tables of 4e6 domains (256 MB) are kept while a graph has them and freed after it."""
    import torch
    N = 4000000
    X = torch.ones((1, N), device="cuda")
    D = torch.empty((1, 2), device="cuda")
    s = torch.cuda.Stream()
    q.qpm_release_caches()
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    g = capture(lambda: q.qpm_eval(N, K1, K2, X, D), s)
    q.qpm_release_caches()
    held = free0 - torch.cuda.mem_get_info()[0]
    assert held > 200e6
    g.replay()
    torch.cuda.synchronize()
    del g
    end = time.monotonic() + 10
    while free0 - torch.cuda.mem_get_info()[0] > held - 200e6 and time.monotonic() < end:
        time.sleep(0.05)  # CUDA tells of a destroyed graph on a thread of its own
        q.qpm_release_caches()
    assert free0 - torch.cuda.mem_get_info()[0] < held - 200e6
