"""The performance cases of this library: what a user's program has it do.

Each case is one call (or one whole design run) through the public Python entry points,
at the sizes of this repository's workloads and benchmark, of the paper's tables, and of
ragged shapes in between.  `listed()` gives the fixed cases, `draw(rng)` more of the same
ranges; `prepare` makes the inputs and plans, `run` is one pass, `work` what a pass cannot
do without, and `exact` the FP64 value of the computed numbers.

A case's "kind" says which path it takes:
  eval    qpm_eval of a float population        packed  qpm_eval_packed of sign words
  multi   qpm_eval_multi (K cascaded problems)  shg     qpm_eval_shg
  adjoint relaxed fitness and its gradient      run     one HWSDA instance, whole run
  design  a multi-wavelength design run         batch   many instances in one launch
"""
import math

import numpy as np
import torch

import paper_2511_01255_gb300 as q
from paper_2511_01255_gb300 import workloads as W

KAPPAS = [(k1, k2) for k1, k2 in W.DESIGN_THG3["kappas"]] + [(W.TWO_PI / 8.0, W.TWO_PI / 1.9)]
K1, K2 = W.PAPER_SCALE["kappa1"], W.PAPER_SCALE["kappa2"]
L2_BYTES = 126e6
MODES = {"launches": q.RUN_LAUNCHES, "graph": q.RUN_GRAPH, "persistent": q.RUN_PERSISTENT}


def listed():
    return [
        # the fitness of one optimiser population (N = 1000 domains, NP = 256) evaluated by a
        # user's own search loop: the smallest call, where latency and launches count
        dict(name="eval_population", kind="eval", N=1000, NP=256, ld=1000, comp=0, k1=K1, k2=K2),
        # bulk evaluation of long crystals (L = 100 mm at 1 um), the precision workload's size
        dict(name="eval_long", kind="eval", N=100000, NP=1024, ld=100000, comp=1, k1=K1, k2=K2),
        # the paper's population of 5000 with an odd crystal length: contiguous rows that do not
        # start on 16-byte boundaries
        dict(name="eval_odd_rows", kind="eval", N=6601, NP=5000, ld=6601, comp=0, k1=K1, k2=K2),
        # the same long crystals kept as packed signs, the form in which designs are stored
        dict(name="packed_long", kind="packed", N=100000, NP=1024, ld=3125, comp=0, k1=K1, k2=K2),
        # the objective of the three-wavelength design evaluated on its whole population
        dict(name="multi_thg3", kind="multi", N=3000, NP=5000, ld=3000, K=3),
        # the SHG field of the five-wavelength design's population (one of its wavelengths)
        dict(name="shg_population", kind="shg", N=3000, NP=5000, ld=3000, k1=W.DESIGN_SHG5["kappas"][0][0]),
        # gradient-based design: the relaxed fitness of a batch and its adjoint (forward and
        # backward into the caller's buffers, as an ascent loop does it)
        dict(name="adjoint_batch", kind="adjoint", B=4096, N=4096, ld=4096, entry="pair", k1=K1, k2=K2),
        # the benchmark's design run: 1000 domains, 256 wolves, 2000 generations
        dict(name="run_paper_scale", kind="run", N=1000, NP=256, G=2000, mode="persistent", comp=1,
             combine=0, fs=0, k1=K1, k2=K2),
        # the middle row of the paper's timing table: NP = 5000, L = 660 um at 0.2 um (N = 3300), with
        # the paper's adaptive F; fewer generations than its 1000
        dict(name="run_table_n3300", kind="run", N=3300, NP=5000, G=200, mode="persistent", comp=0,
             combine=0, fs=2, k1=K1, k2=K2),
        # the precision workload: 1e5 domains, 1024 wolves, compensated sums
        dict(name="run_long", kind="run", N=100000, NP=1024, G=100, mode="persistent", comp=1,
             combine=0, fs=0, k1=K1, k2=K2),
        # the three-wavelength design of Sec. 5 (N = 3000, NP = 5000), the autotuned team width
        dict(name="design_thg3", kind="design", obj="thg", N=3000, NP=5000, G=200, K=3, team=64,
             mode="launches", fs=0),
        # a parameter study: 512 independent instances of uneven size in one launch
        dict(name="batch_512", kind="batch", n=512, sizes=1, G=100, cluster=2),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _kappa(rng):
    return W.TWO_PI / rng.uniform(6.0, 8.0), W.TWO_PI / rng.uniform(1.3, 2.0)


def _ld(rng, N):
    """Contiguous rows, rows padded to 16 bytes, or a slice of a wider array."""
    return rng.choice([N, N, (N + 3) // 4 * 4, N + rng.randrange(1, 64)])


def draw(rng):
    kind = rng.choice(["eval", "eval", "packed", "multi", "shg", "adjoint", "adjoint", "run", "run", "run",
                       "design", "batch"])
    k1, k2 = _kappa(rng)
    if kind in ("eval", "packed"):
        N = _log(rng, 500, 100000)
        NP = _log(rng, 32, min(8192, 102400000 // N))
        W32 = (N + 31) // 32
        ld = _ld(rng, N) if kind == "eval" else rng.choice([W32, (W32 + 3) // 4 * 4])
        return dict(kind=kind, N=N, NP=NP, ld=ld, comp=rng.randrange(2), k1=k1, k2=k2)
    if kind in ("multi", "shg"):
        N = _log(rng, 500, 13200)
        NP = _log(rng, 64, min(5000, 33000000 // N))
        if kind == "shg":
            return dict(kind=kind, N=N, NP=NP, ld=_ld(rng, N), k1=W.TWO_PI / rng.uniform(2.0, 5.0))
        return dict(kind=kind, N=N, NP=NP, ld=_ld(rng, N), K=rng.randrange(1, 5))
    if kind == "adjoint":
        N = _log(rng, 64, 8192)
        entry = rng.choice(["pair", "autograd"])
        return dict(kind=kind, B=_log(rng, 3, min(8192, 16777216 // N)), N=N,
                    ld=N if entry == "autograd" else _ld(rng, N), entry=entry, k1=k1, k2=k2)
    if kind == "run":
        if rng.random() < 0.25:
            N, NP = _log(rng, 13200, 100000), _log(rng, 64, 1024)
        else:
            N, NP = _log(rng, 500, 13200), _log(rng, 64, 5000)
        combine = rng.choice([0, 0, 1, 2])
        mode = rng.choice(["launches", "graph"] if combine == 2 else ["persistent", "persistent", "graph"])
        G = max(10, min(1000, int(3.0e9 / (N * NP))))
        return dict(kind=kind, N=N, NP=NP, G=G, mode=mode, comp=rng.randrange(2), combine=combine,
                    fs=rng.randrange(3), k1=k1, k2=k2)
    if kind == "design":
        obj = rng.choice(["thg", "shg"])
        N, NP = _log(rng, 500, 4000), _log(rng, 256, 5000)
        return dict(kind=kind, obj=obj, N=N, NP=NP, G=max(20, min(200, int(3.0e9 / (N * NP)))),
                    K=rng.randrange(2, 5 if obj == "thg" else 6), team=rng.choice([0, 32, 64, 128]),
                    mode=rng.choice(["launches", "graph"]), fs=rng.randrange(3))
    n = _log(rng, 32, 512)
    return dict(kind="batch", n=n, sizes=rng.randrange(1, 1000), G=max(10, min(100, 25000 // n)),
                cluster=rng.choice([1, 2, 4]))


# ------------------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _genes(NP, N, ld, k1, k2, seed):
    """float32 [NP, N] (leading dimension ld): the signs of a two-tone design, each row with
    its own share of flipped domains from 0 (a converged wolf) to 1/2 (a random one),
    magnitudes U(0, 1)."""
    g = _gen(seed)
    base = torch.from_numpy(W.two_tone_signs(N, k1, k2)).cuda()
    buf = torch.zeros((NP, ld), dtype=torch.float32, device="cuda")
    share = torch.linspace(0.0, 0.5, NP, device="cuda")
    for r in range(0, NP, 256):
        e = min(NP, r + 256)
        flip = torch.rand((e - r, N), generator=g, device="cuda") < share[r:e, None]
        mag = torch.rand((e - r, N), generator=g, device="cuda").clamp_(min=1e-6)
        buf[r:e, :N] = torch.where(flip, -base, base) * mag
    return buf[:, :N] if ld != N else buf


def _signs(NP, N, ld, k1, k2, seed):
    words = torch.zeros((NP, ld), dtype=torch.int32, device="cuda")
    W32 = (N + 31) // 32
    bit = torch.arange(32, device="cuda", dtype=torch.int64)
    for r in range(0, NP, 128):
        e = min(NP, r + 128)
        neg = torch.zeros((e - r, W32 * 32), dtype=torch.int64, device="cuda")
        # every chunk from its own seed: the whole float population is never held
        share = torch.linspace(0.0, 0.5, NP, device="cuda")[r:e, None]
        base = torch.from_numpy(W.two_tone_signs(N, k1, k2)).cuda()
        flip = torch.rand((e - r, N), generator=_gen(int(seed) * 1000003 + r), device="cuda") < share
        neg[:, :N] = (torch.where(flip, -base, base) < 0).to(torch.int64)
        w = (neg.view(e - r, W32, 32) << bit).sum(2)
        words[r:e, :W32] = torch.where(w >= 1 << 31, w - (1 << 32), w).to(torch.int32)
    return words


def _theta(c, seed):
    """theta float32 [B, N]: N(0, 1) around designs of strength 0 (the random start) to 2."""
    g = _gen(seed)
    base = torch.from_numpy(W.two_tone_signs(c["N"], c["k1"], c["k2"])).cuda()
    buf = torch.zeros((c["B"], c["ld"]), dtype=torch.float32, device="cuda")
    buf[:, :c["N"]] = torch.randn((c["B"], c["N"]), generator=g, device="cuda")
    buf[:, :c["N"]] += torch.linspace(0.0, 2.0, c["B"], device="cuda")[:, None] * base
    gf = torch.rand(c["B"], generator=g, device="cuda") + 0.5
    return (buf[:, :c["N"]] if c["ld"] != c["N"] else buf), gf


def _objective(c):
    if c["obj"] == "thg":
        return W.DESIGN_THG3["kind"], KAPPAS[:c["K"]], 2.0 / 9.0 * c["N"] ** 2, 0.5
    return W.DESIGN_SHG5["kind"], W.DESIGN_SHG5["kappas"][:c["K"]], 2.0 / 3.0 * c["N"], 0.5


def prepare(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind in ("eval", "packed"):
        make = _genes if kind == "eval" else _signs
        X = make(c["NP"], c["N"], c["ld"], c["k1"], c["k2"], seed)
        return dict(c=c, X=X, D=torch.empty((c["NP"], 2), device="cuda"), f=torch.empty(c["NP"], device="cuda"))
    if kind == "multi":
        X = _genes(c["NP"], c["N"], c["ld"], *KAPPAS[0], seed)
        return dict(c=c, X=X, D=torch.empty((c["NP"], c["K"], 2), device="cuda"),
                    f=torch.empty(c["NP"], device="cuda"))
    if kind == "shg":
        X = _genes(c["NP"], c["N"], c["ld"], c["k1"], c["k1"], seed)
        return dict(c=c, X=X, D=torch.empty((c["NP"], 2), device="cuda"), f=torch.empty(c["NP"], device="cuda"))
    if kind == "adjoint":
        theta, gf = _theta(c, seed)
        s = dict(c=c, theta=theta, gf=gf)
        if c["entry"] == "pair":
            s.update(D=torch.empty((c["B"], 2), device="cuda"), f=torch.empty(c["B"], device="cuda"),
                     saved=q.relaxed_saved(c["B"], c["N"]), grad=torch.empty((c["B"], c["N"]), device="cuda"))
        else:
            theta.requires_grad_(True)
        return s
    seed = int(seed) & 0xFFFFFFFF
    if kind == "run":
        prm = q.Params(c["NP"], c["G"], 0.5, 0.9, seed, c["combine"], c["comp"], 0, c["fs"])
        return dict(c=c, st=q.State([(c["N"], c["k1"], c["k2"])], [prm]))
    if kind == "design":
        obj, kappas, G0, beta = _objective(c)
        prm = q.Params(c["NP"], c["G"], 0.5, 0.9, seed, 0, 0, c["team"], c["fs"])
        st = q.State([(c["N"], *kappas[0])], [prm])
        st.set_objective(obj, kappas, G0, beta)
        return dict(c=c, st=st)
    inst = W.batched_instances(c["n"], seed=c["sizes"])
    st = q.State([(i["N"], i["kappa1"], i["kappa2"]) for i in inst],
                 [q.Params(i["NP"], c["G"], i["F"], i["CR"], seed, 0, i["compensated"], 0, 0) for i in inst])
    st.set_batch_cluster(c["cluster"])
    rows, cols = np.array([i["NP"] for i in inst]), np.array([i["N"] for i in inst])
    up = (cols + 3) // 4 * 4  # the best genes of every instance start on 16 bytes
    return dict(c=c, st=st, inst=inst,
                pop=torch.zeros(int((rows * cols).sum()), device="cuda"), fit=torch.zeros(int(rows.sum()), device="cuda"),
                best=torch.zeros(int(up.sum()), device="cuda"),
                d64=torch.zeros((c["n"], 2), dtype=torch.float64, device="cuda"),
                bfit=torch.zeros(c["n"], device="cuda"), idx=torch.zeros(c["n"], dtype=torch.int32, device="cuda"))


# ------------------------------------------------------------------------------ one pass
def run(s):
    c = s["c"]
    kind = c["kind"]
    if kind == "eval":
        q.qpm_eval(c["N"], c["k1"], c["k2"], s["X"], s["D"], s["f"], c["comp"])
        return dict(D=s["D"], f=s["f"])
    if kind == "packed":
        q.qpm_eval_packed(c["N"], c["k1"], c["k2"], s["X"], s["D"], s["f"], c["comp"])
        return dict(D=s["D"], f=s["f"])
    if kind == "multi":
        _, _, G0, beta = _objective(dict(c, obj="thg"))
        q.qpm_eval_multi(c["N"], KAPPAS[:c["K"]], s["X"], G0, beta, s["f"], s["D"])
        return dict(D=s["D"], f=s["f"])
    if kind == "shg":
        q.qpm_eval_shg(c["N"], c["k1"], s["X"], s["D"], s["f"])
        return dict(D=s["D"], f=s["f"])
    if kind == "adjoint":
        if c["entry"] == "autograd":
            f = q.deff_relaxed(s["theta"], c["k1"], c["k2"])
            grad, = torch.autograd.grad(f, s["theta"], s["gf"])
            return dict(f=f.detach(), grad=grad)
        q.qpm_deff_relaxed_fwd(c["N"], c["k1"], c["k2"], s["theta"], s["D"], s["f"], s["saved"])
        q.qpm_deff_relaxed_bwd(c["N"], c["k1"], c["k2"], s["theta"], s["D"], s["saved"], s["gf"], s["grad"])
        return dict(D=s["D"], f=s["f"], grad=s["grad"])
    st = s["st"]
    st.init()
    if kind in ("run", "design"):  # the whole run, then its best design and its population
        st.run(c["G"], MODES[c["mode"]])
        x, d64, f, idx = st.best()
        X, fit, D = st.population()
        return dict(best=x, d64=d64, best_f=f, index=idx, genes=X, fit=fit, D=D)
    st.run(c["G"], q.RUN_BATCHED)
    a = b = e = 0
    for k, i in enumerate(s["inst"]):  # every instance's best design and population
        N, NP = i["N"], i["NP"]
        q.qpm_get_best(st.h, k, s["best"][e:e + N], s["d64"][k], s["bfit"][k:k + 1], s["idx"][k:k + 1])
        q.qpm_get_population(st.h, k, s["pop"][a:a + N * NP].view(NP, N), s["fit"][b:b + NP])
        a, b, e = a + N * NP, b + NP, e + (N + 3) // 4 * 4
    return dict(best=s["best"], d64=s["d64"], best_f=s["bfit"], index=s["idx"], genes=s["pop"], fit=s["fit"])


# ------------------------------------------------------------------------------ the work
def _search_work(N, NP, G, scans):
    """One HWSDA run: the population is written out once; one that does not fit the L2 cache
    is read and written once more in each phase of each generation.  FP32 operations of a
    gene and generation: 3 (DE) + 23 (three leaders' pulls and their mean) + two evaluations
    of 12 per cascaded scan (complex multiply-add and two running sums)."""
    pop = 4.0 * N * NP
    return {"bytes": pop + (4 * pop * G if 2 * pop > L2_BYTES else 0), "flops": (26.0 + 2 * scans) * N * NP * G}


def work(case):
    c = case
    kind = c["kind"]
    if kind in ("eval", "packed"):
        row = 4 * c["N"] if kind == "eval" else 4 * ((c["N"] + 31) // 32)
        return {"bytes": c["NP"] * (row + 12.0), "flops": 12.0 * c["N"] * c["NP"]}
    if kind == "multi":
        return {"bytes": c["NP"] * (4.0 * c["N"] + 8 * c["K"] + 4), "flops": 12.0 * c["K"] * c["N"] * c["NP"]}
    if kind == "shg":
        return {"bytes": c["NP"] * (4.0 * c["N"] + 12), "flops": 4.0 * c["N"] * c["NP"]}
    if kind == "adjoint":  # theta read and the gradient written, once each
        return {"bytes": c["B"] * (8.0 * c["N"] + 16), "flops": 60.0 * c["N"] * c["B"]}
    if kind == "run":
        return _search_work(c["N"], c["NP"], c["G"], 12)
    if kind == "design":
        return _search_work(c["N"], c["NP"], c["G"], c["K"] * (12 if c["obj"] == "thg" else 4))
    parts = [_search_work(i["N"], i["NP"], c["G"], 12) for i in W.batched_instances(c["n"], seed=c["sizes"])]
    genes = sum(4.0 * i["N"] * i["NP"] for i in W.batched_instances(c["n"], seed=c["sizes"]))
    # the instances' populations together do not fit the L2 cache
    return {"bytes": genes + (4 * genes * c["G"] if 2 * genes > L2_BYTES else 0), "flops": sum(p["flops"] for p in parts)}


# ------------------------------------------------------------------------------ FP64 values
def _phi(k):
    return (1 - np.exp(-1j * k)) / (1j * k)


def _consts(k1, k2):
    return complex(_phi(k1) * _phi(k2)), complex((_phi(k2) - _phi(k1 + k2)) / (1j * k1))


def _phasors(N, k):
    return torch.exp(-1j * k * torch.arange(N, dtype=torch.float64, device="cuda"))


def _chunks(rows, N):
    step = max(1, 16000000 // N)
    return [(r, min(rows, r + step)) for r in range(0, rows, step)]


def _field(d, k1, k2):
    """d_eff of rows of real domain values d (float64 [rows, N]), complex128 [rows]."""
    p1, p2 = _phasors(d.shape[1], k1), _phasors(d.shape[1], k2)
    phi12, psi = _consts(k1, k2)
    b = d * p1
    pre = torch.cumsum(b, 1) - b
    return phi12 * (d * p2 * pre).sum(1) + psi * (d * d * (p1 * p2)).sum(1)


def _pm(x):
    one = torch.ones((), dtype=torch.float64, device="cuda")
    return torch.where(x < 0, -one, one)


def _unpack(words, N):
    bit = torch.arange(32, device="cuda", dtype=torch.int32)
    neg = (words[:, :, None] >> bit) & 1
    return 1.0 - 2.0 * neg.view(words.shape[0], -1)[:, :N].to(torch.float64)


def exact(case, seed):
    c = case
    kind = c["kind"]
    if kind in ("run", "design", "batch"):
        return None  # thousands of dependent random decisions: no value but the run's own
    s = prepare(case, seed)
    if kind == "adjoint":
        th = s["theta"].detach()
        f, D, grad = [], [], []
        k1, k2 = c["k1"], c["k2"]
        p1, p2 = _phasors(c["N"], k1), _phasors(c["N"], k2)
        phi12, psi = _consts(k1, k2)
        for r, e in _chunks(c["B"], 4 * c["N"]):
            d = torch.tanh(th[r:e].double())
            Dc = _field(d, k1, k2)
            b, a = d * p1, d * p2
            pre = torch.cumsum(b, 1) - b
            suf = a.sum(1, keepdim=True) - torch.cumsum(a, 1)
            dD = phi12 * (p2 * pre + p1 * suf) + 2 * psi * d * (p1 * p2)
            g = 2 * (Dc.conj()[:, None] * dD).real * (1 / torch.cosh(th[r:e].double())) ** 2
            f.append(Dc.abs() ** 2)
            D.append(torch.view_as_real(Dc))
            grad.append(g * s["gf"][r:e, None].double())
        out = dict(f=torch.cat(f), grad=torch.cat(grad))
        if c["entry"] == "pair":
            out["D"] = torch.cat(D)
        return out
    D = []
    for r, e in _chunks(c["NP"], c["N"]):
        d = _unpack(s["X"][r:e, :(c["N"] + 31) // 32], c["N"]) if kind == "packed" else _pm(s["X"][r:e])
        if kind == "multi":
            D.append(torch.stack([_field(d, k1, k2) for k1, k2 in KAPPAS[:c["K"]]], 1))
        elif kind == "shg":
            D.append(complex(_phi(c["k1"])) * (d * _phasors(c["N"], c["k1"])).sum(1))
        else:
            D.append(_field(d, c["k1"], c["k2"]))
    D = torch.cat(D)
    if kind == "multi":
        _, _, G0, beta = _objective(dict(c, obj="thg"))
        G = D.abs()
        f = (float(np.float32(G0)) - G).abs().sum(1) + beta * (G.max(1).values - G.min(1).values)
        return dict(D=torch.view_as_real(D), f=f)
    return dict(D=torch.view_as_real(D), f=D.abs() ** 2)
