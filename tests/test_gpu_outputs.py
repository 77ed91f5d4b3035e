"""GPU parity of a state's outputs: the population in natural order and the best design.

qpm_get_population returns the genes qpm_set_population was given bit for bit, whatever
the rows' permutation (team width, domains per thread) and the output rows' alignment;
qpm_get_best returns the row of the largest fitness (lowest index on ties) and its FP64
d_eff within 1e-9 of the oracle (the scale floor of helpers.deff_err).
"""
import math

import numpy as np
import pytest

from helpers import deff_err

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


# team 32: c = 4 ceil(N / 128) domains per thread (1, 2, 3, 5 and 16 groups: runs of 1 to 8 and a
# second tile); wider teams: one group per thread and several; N on both sides of 128
@pytest.mark.parametrize("N,team", [(1, 32), (127, 32), (128, 32), (129, 32), (257, 32), (520, 32),
                                    (2001, 32), (1000, 256), (3300, 256), (5003, 512)])
@pytest.mark.parametrize("ld_extra", [0, 1, 4])
def test_population_and_best(q, orc, N, team, ld_extra):
    import torch
    NP, ld = 9, (N + ld_extra if ld_extra != 4 else (N + 3) // 4 * 4 + 4)
    rng = np.random.default_rng(N + team + ld_extra)
    X = rng.uniform(-1, 1, (NP, N)).astype(np.float32)
    X[6] = X[2]  # a tie
    with q.State([(N, K1, K2)], [q.Params(NP, 3, 0.5, 0.9, 5, 0, 0, team, 0)]) as st:
        st.init()
        q.qpm_set_population(st.h, 0, torch.from_numpy(X).cuda(), 0)
        buf = torch.full((NP, ld), 7.0, device="cuda")
        f, D = torch.empty(NP, device="cuda"), torch.empty((NP, 2), device="cuda")
        q.qpm_get_population(st.h, 0, buf[:, :N], f, D)
        x, d64, fb, idx = st.best()
        out = buf.cpu().numpy()
    assert np.array_equal(out[:, :N], X)
    assert (out[:, N:] == 7.0).all()  # nothing past a row's N genes is written
    f = f.cpu().numpy()
    i = int(idx.item())
    assert i == int(np.argmax(f)) and fb.item() == f[i]
    assert np.array_equal(x.cpu().numpy(), X[i])
    ref = orc.deff_genes(X[i:i + 1], K1, K2)
    assert deff_err(d64.cpu().numpy()[None], ref, N).max() < 1e-9


def test_many_instances_start_like_single_launches(q):
    """The initialisation of many instances in one launch: the same tables, populations and
    fitness as the launch per instance (a state whose teams are wider than a warp) gives for
    rows short enough that both sum in the same order (one domain group per thread)."""
    import torch
    sizes = [(N, NP) for N, NP in [(100, 5), (128, 64), (3, 4), (90, 33)]]
    probs = [(N, K1 + 0.01 * k, K2) for k, (N, _) in enumerate(sizes)]
    prms = [q.Params(NP, 2, 0.5, 0.9, 3, 0, k % 2, 32, 0) for k, (_, NP) in enumerate(sizes)]
    with q.State(probs, prms) as st:
        st.init()
        got = [[a.clone() for a in st.population(k)] for k in range(4)]
    # a fifth instance of another width sends every instance down the launch per instance
    with q.State(probs + [(64, K1, K2)], prms + [q.Params(8, 2, 0.5, 0.9, 3, 0, 0, 64, 0)]) as st:
        st.init()
        for k in range(4):
            for a, b in zip(got[k], st.population(k)):
                assert torch.equal(a, b)


@pytest.mark.parametrize("sizes", [[(100, 5), (257, 64), (1000, 7), (3300, 33)], [(8000, 4), (129, 70)]])
def test_many_instances_of_mixed_sizes_start_like_single_launches(q, sizes):
    """Tables of several and of unequal numbers of CTAs, several domain groups per thread."""
    import torch
    n = len(sizes)
    probs = [(N, K1 + 0.01 * k, K2) for k, (N, _) in enumerate(sizes)]
    prms = [q.Params(NP, 2, 0.5, 0.9, 3 + k, 0, k % 2, 32, 0) for k, (_, NP) in enumerate(sizes)]
    with q.State(probs, prms) as st:
        st.init()
        got = [[a.clone() for a in st.population(k) + st.best(k)] for k in range(n)]
    with q.State(probs + [(64, K1, K2)], prms + [q.Params(8, 2, 0.5, 0.9, 3, 0, 0, 64, 0)]) as st:
        st.init()
        for k in range(n):
            for a, b in zip(got[k], st.population(k) + st.best(k)):
                assert torch.equal(a, b)
