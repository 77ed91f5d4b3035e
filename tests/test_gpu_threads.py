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
