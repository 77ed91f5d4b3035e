"""GPU parity of the row sweeps at the edges of their splits, against the oracle's FP64 scan.

Rows of every alignment (the four classes of a pitch that is no multiple of 16 bytes, bases 0
to 3 floats off), populations around the 32-row groups and the row blocks of a CTA, lengths
around the 4-domain blocks, 32-domain tiles, 128-domain table steps and the longest run, rows
combined by the sweep itself and by the combining kernel.  Genes include -0.0 (counts as +1).
"""
import math

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


def rows_of(NP, N, ld, off, seed):
    """(torch view [NP, N] with leading dimension ld, `off` floats into its buffer; numpy genes)"""
    import torch
    rng = np.random.default_rng(seed)
    X = rng.uniform(-1, 1, (NP, N)).astype(np.float32)
    X[rng.random((NP, N)) < 0.02] = -0.0
    flat = torch.full((off + (NP - 1) * ld + N,), -9.0)  # ends with the last row's last gene
    flat = flat.cuda()
    view = flat[off:].as_strided((NP, N), (ld, 1))
    view.copy_(torch.from_numpy(X))
    return view, X


SHAPES = [(1, 1, 1, 1), (3, 2, 5, 0), (31, 5, 31, 3), (33, 33, 33, 0), (64, 4, 64, 2), (127, 7, 130, 1),
          (128, 130, 128, 0), (129, 129, 129, 1), (1000, 256, 1000, 0), (1921, 32, 1921, 0),
          (1923, 40, 1924, 2), (5003, 161, 5003, 3), (777, 700, 777, 0), (30011, 3, 30011, 1)]


@pytest.mark.parametrize("N,NP,ld,off", SHAPES)
@pytest.mark.parametrize("comp", [0, 1])
def test_float_rows(q, orc, N, NP, ld, off, comp):
    import torch
    view, X = rows_of(NP, N, ld, off, N + NP)
    D, f = torch.empty((NP, 2), device="cuda"), torch.empty(NP, device="cuda")
    for _ in range(2):  # the second call finds the counters of the first
        D.fill_(float("nan"))
        q.qpm_eval(N, K1, K2, view, D, f, comp)
    D = D.cpu().numpy()
    ref = orc.deff_closed_genes(X, K1, K2)
    assert deff_err(D, ref, N).max() < TOL_D
    assert np.allclose(f.cpu().numpy(), (D.astype(np.float64) ** 2).sum(1), rtol=1e-6)


@pytest.mark.parametrize("N,NP", [(1, 1), (31, 33), (97, 64), (128, 65), (129, 300), (4097, 257), (30001, 5)])
@pytest.mark.parametrize("pad,comp", [(0, 0), (1, 1)])
def test_packed_rows(q, orc, N, NP, pad, comp):
    import torch
    from paper_2511_01255_gb300 import workloads as W
    X = W.random_genes(NP, N, seed=N + NP)
    words = W.pack_signs(X, N)
    ld = (words.shape[1] + 3) // 4 * 4 if pad else words.shape[1]
    flat = torch.zeros((NP, ld), dtype=torch.int32, device="cuda")
    flat[:, :words.shape[1]] = torch.from_numpy(words.view(np.int32)).cuda()
    D = torch.empty((NP, 2), device="cuda")
    q.qpm_eval_packed(N, K1, K2, flat, D, None, comp)
    assert deff_err(D.cpu().numpy(), orc.deff_closed_genes(X, K1, K2), N).max() < TOL_D


@pytest.mark.parametrize("K", [1, 2, 3, 4])
@pytest.mark.parametrize("N,NP,ld,off", [(5, 3, 7, 1), (130, 33, 130, 0), (1000, 300, 1000, 0),
                                         (1001, 261, 1001, 2), (30001, 9, 30001, 0)])
def test_multi_rows(q, orc, K, N, NP, ld, off):
    import torch
    view, X = rows_of(NP, N, ld, off, K + N)
    kap = [(K1 + 0.05 * k, K2 - 0.1 * k) for k in range(K)]
    G0, beta = 0.2 * N * N, 0.5
    D, f = torch.empty((NP, K, 2), device="cuda"), torch.empty(NP, device="cuda")
    q.qpm_eval_multi(N, kap, view, G0, beta, f, D)
    ref = np.stack([orc.deff_closed_genes(X, *k) for k in kap], 1)
    D = D.cpu().numpy()
    for k in range(K):
        assert deff_err(D[:, k], ref[:, k], N).max() < TOL_D
    G = np.abs(ref)
    obj = np.abs(G0 - G).sum(1) + beta * (G.max(1) - G.min(1))
    assert np.abs(f.cpu().numpy() - obj).max() <= TOL_D * K * max(G0, N * N / 2)


@pytest.mark.parametrize("N", [1, 3, 4, 5, 127, 255, 256, 257, 511, 515])
@pytest.mark.parametrize("NP,pad,off", [(1, 0, 0), (4, 1, 0), (153, 0, 1), (609, 0, 0)])
def test_shg_rows(q, orc, N, NP, pad, off):
    import torch
    view, X = rows_of(NP, N, (N + 3) // 4 * 4 if pad else N, off, 3 * N + NP)
    E = torch.empty((NP, 2), device="cuda")
    q.qpm_eval_shg(N, K1, view, E)
    E = E.cpu().numpy()
    ref = orc.shg_genes(X, K1)
    # random rows cancel: floor at 1e-3 of the all-up magnitude scale N
    assert (np.abs(E[:, 0] + 1j * E[:, 1] - ref) / np.maximum(np.abs(ref), 1e-3 * N)).max() < TOL_D


# A captured call leaves the rows to the combining kernel, which takes the same tree over up to 16
# pieces: the same bits as the sweep's own combination.
@pytest.mark.parametrize("N,NP,K", [(129, 129, 1), (1000, 256, 1), (1923, 40, 1), (5003, 2100, 1),
                                    (1000, 256, 2), (5003, 2100, 3)])
def test_captured_rows_same_bits(q, N, NP, K):
    import torch
    view, _ = rows_of(NP, N, N, 0, N + K)
    kaps = [(K1 * (1 + 0.01 * k), K2) for k in range(K)]
    D = torch.empty((NP, 2 * K), device="cuda")
    f = torch.empty(NP, device="cuda")
    s = torch.cuda.Stream()

    def call():
        if K == 1:
            q.qpm_eval(N, K1, K2, view, D, f, 1)
        else:
            q.qpm_eval_multi(N, kaps, view, 1e5, 0.5, f, D)

    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        call()  # tables and the stream's scratch
        s.synchronize()
        call()  # sees the tables complete
        s.synchronize()
        ref = D.clone()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        call()
    for _ in range(2):
        D.fill_(float("nan"))
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(D, ref)


# up to as many rows as SMs a CTA has one row; from 64 rows per CTA on it keeps its sums in passes
@pytest.mark.parametrize("NP", ["sms", "sms+1", "64sms+5"])
@pytest.mark.parametrize("N,off", [(260, 0), (259, 1), (1030, 0)])
def test_shg_rows_per_cta(q, orc, NP, N, off):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    NP = {"sms": sms, "sms+1": sms + 1, "64sms+5": 64 * sms + 5}[NP]
    view, X = rows_of(NP, N, N, off, N + NP)
    E, f = torch.full((NP, 2), float("nan"), device="cuda"), torch.empty(NP, device="cuda")
    q.qpm_eval_shg(N, K1, view, E, f)
    E = E.cpu().numpy()
    ref = orc.shg_genes(X, K1)
    assert (np.abs(E[:, 0] + 1j * E[:, 1] - ref) / np.maximum(np.abs(ref), 1e-3 * N)).max() < TOL_D


# few row blocks of rows long enough for three rounds of CTAs: aligned rows take runs of the full
# length instead, rows of odd pitch whole rounds; K = 1 of the multi-wavelength call splits alike
@pytest.mark.parametrize("N,NP,ld", [(2900000, 33, 2900000), (2900000, 33, 2900001)])
def test_long_rows(q, orc, N, NP, ld):
    import torch
    buf = torch.empty((NP, ld), device="cuda").uniform_(-1, 1, generator=torch.Generator("cuda").manual_seed(5))
    X = buf[:, :N]
    D, M, f = (torch.full(s, float("nan"), device="cuda") for s in ((NP, 2), (NP, 1, 2), (NP,)))
    q.qpm_eval(N, K1, K2, X, D)
    q.qpm_eval_multi(N, [(K1, K2)], X, 1e5, 0.5, f, M)
    torch.cuda.synchronize()
    assert torch.equal(D, M[:, 0])
    rows = [0, 31, 32]
    ref = orc.deff_closed_genes(X[rows].cpu().numpy(), K1, K2)
    assert deff_err(D[rows].cpu().numpy(), ref, N).max() < TOL_D
