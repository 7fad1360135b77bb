"""The work that users of this library have it do, as cases to time.

Six kinds of call, each through the public binding (pcomp) on seeded
synthetic instances (workloads):

* ``sqa``    DT-SQA anneals of one lattice instance: pc_sqa_anneal, or
             pc_sqa_setup_bc + pc_sqa_run with open axes or final spins;
* ``apt``    a stretch of APT(+ICM) on a loaded batch of lattices: pc_apt_run,
             then the best energies, their hit sweeps and the best states;
* ``gapt``   the same on general graphs: pc_gapt_run, then the best states;
* ``gsqa``   DT-SQA of one general graph: pc_gsqa_anneal;
* ``ladder`` the adaptive ladders of a batch: pc_adaptive_ladder;
* ``mlp``    training steps of the ladder network: pc_mlp_train_step_dev.

A case is a dict of plain values; ``listed`` names twelve and ``draw`` gives
more of the same ranges.
"""
import math

import numpy as np
import torch

from paper_2503_10302_gb300 import pcomp
from paper_2503_10302_gb300 import workloads as W

# 32-bit integer operations of one spin update in the plain per-site form: a
# quarter of a Philox4x32-10 call (10), the six-neighbour field (6), table
# index, lookup, compare and store (4).
OPS_PER_UPDATE = 20
SQA_T = 0.05            # temperature of every anneal
GAP_WEIGHT = 0.05       # relative-gap term of the ladder network's loss


def listed():
    return [
        # a first look at a small instance: few runs, few sweeps, final spins
        dict(name="sqa_small", kind="sqa", lx=4, ly=4, lz=4, open_xy=False, P=16, R=8, sweeps=100, spins=True),
        # the headline anneal: 512 spins, 64 slices, 256 runs, 10^4 sweeps
        dict(name="sqa_8x64x256", kind="sqa", lx=8, ly=8, lz=8, open_xy=False, P=64, R=256, sweeps=10000,
             spins=False),
        # the paper's 15 x 15 x 12 shape, open in x and y (padded to even lengths with vacancies), R = 132
        dict(name="sqa_15x15x12_open", kind="sqa", lx=15, ly=15, lz=12, open_xy=True, P=64, R=132, sweeps=1000,
             spins=False),
        # one small instance, 8 temperatures x 2 labels: a single CTA's latency
        dict(name="apt_L4", kind="apt", n=1, lx=4, ly=4, lz=4, sizes="", open_xy=False, T=8, T_min=8, labels=2,
             spp=1, attempts=1000, icm=True, state=True),
        # time-to-target runs of 64 instances of L = 12: ICM and a swap attempt after every sweep
        dict(name="apt_64xL12", kind="apt", n=64, lx=12, ly=12, lz=12, sizes="", open_xy=False, T=32, T_min=32,
             labels=2, spp=1, attempts=1024, icm=True, state=False),
        # the paper's APT setting: 15 x 15 x 12 open in x and y, 32 temperatures x 4 labels
        dict(name="apt_15x15x12_4labels", kind="apt", n=8, lx=15, ly=15, lz=12, sizes="", open_xy=True, T=32,
             T_min=32, labels=4, spp=1, attempts=256, icm=True, state=False),
        # a batch of 256 instances of uneven size, 24-32 temperatures x 2 labels
        dict(name="apt_mixed256", kind="apt", n=256, lx=0, ly=0, lz=0, sizes="6,8,10,12,14,16", open_xy=False, T=32,
             T_min=24, labels=2, spp=1, attempts=512, icm=True, state=False),
        # long best-energy runs of the largest lattices: a swap attempt and ICM every 10 sweeps
        dict(name="apt_128xL16_every10", kind="apt", n=128, lx=16, ly=16, lz=16, sizes="", open_xy=False, T=32,
             T_min=32, labels=2, spp=10, attempts=100, icm=True, state=False),
        # APT + ICM on embedded instances: 64 dimer embeddings of L = 8 (1024 p-bits, 4 colours)
        dict(name="gapt_64xdimerL8", kind="gapt", n=64, graph="dimer", lx=8, ly=8, lz=8, wmax=1, hmax=0, T=32,
             labels=2, spp=1, attempts=512, icm=True),
        # DT-SQA on one embedded instance: dimer embedding of 15 x 15 x 12 (5400 p-bits), 256 runs
        dict(name="gsqa_dimer15x15x12", kind="gsqa", graph="dimer", lx=15, ly=15, lz=12, wmax=1, P=64, R=256,
             sweeps=200),
        # the adaptive ladders that the 64 x L = 12 runs start with
        dict(name="ladder_64xL12", kind="ladder", n=64, L=12, chains=32, sweeps=2000, tail=500),
        # training of the ladder network: 10 minibatches of 256
        dict(name="mlp_256x10", kind="mlp", batch=256, steps=10),
    ]


def _log(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["sqa", "sqa", "apt", "apt", "apt", "gapt", "gsqa", "ladder", "mlp"])
    if kind == "sqa":
        open_xy = rng.random() < 0.4
        if open_xy:   # odd lengths are allowed on the open axes
            lx, ly, lz = rng.randint(3, 15), rng.randint(3, 15), 2 * rng.randint(2, 6)
        else:
            lx, ly, lz = (2 * rng.randint(1, 6) for _ in range(3))
        P = 16 * rng.randint(1, 8)
        n = (lx + lx % 2) * (ly + ly % 2) * lz
        while n * P > 262144:
            P -= 16
        R = _log(rng, 1, 512)
        sweeps = max(3, min(_log(rng, 20, 5000), int(2e10 / (n * P * max(R, 64)))))
        return dict(kind="sqa", lx=lx, ly=ly, lz=lz, open_xy=open_xy, P=P, R=R, sweeps=sweeps,
                    spins=n * P * R <= 1 << 22 and rng.random() < 0.5)
    if kind == "apt":
        mixed = rng.random() < 0.25
        open_xy = (not mixed) and rng.random() < 0.3
        labels = rng.choice([1, 2, 2, 2, 4])
        T = rng.randint(9, 32) if labels == 4 else rng.randint(3, 32)
        if mixed:
            lx = ly = lz = 0
            n, side = _log(rng, 8, 200), 16
        else:
            if open_xy:
                lx, ly, lz = rng.randint(3, 15), rng.randint(3, 15), 2 * rng.randint(2, 6)
            else:
                lx, ly, lz = (2 * rng.randint(2, 8) for _ in range(3))
            n, side = _log(rng, 1, 160), max(lx, ly, lz)
        spp = rng.choice([1, 1, 1, 2, 10])
        attempts = max(5, min(_log(rng, 20, 600), 600 // spp, int(600 * 16 / side / labels)))
        return dict(kind="apt", n=n, lx=lx, ly=ly, lz=lz, sizes="6,8,10,12,14,16" if mixed else "", open_xy=open_xy,
                    T=T, T_min=rng.randint(max(3, T - 8), T) if mixed and labels < 4 else T, labels=labels, spp=spp,
                    attempts=attempts, icm=labels > 1 and rng.random() < 0.75, state=n <= 2)
    if kind == "gapt":
        graph = rng.choice(["dimer", "lattice", "random"])
        if graph == "random":
            lx, ly, lz, wmax = _log(rng, 40, 2000), 1, 1, rng.randint(1, 3)
        elif graph == "lattice":
            lx, ly, lz, wmax = rng.randint(3, 13), rng.randint(3, 13), rng.randint(3, 12), 1
        else:
            lx, ly, lz, wmax = rng.randint(3, 8), rng.randint(3, 8), rng.randint(3, 8), 1
        hmax = rng.choice([0, 0, 2])
        labels = rng.choice([1, 2, 2, 4])
        return dict(kind="gapt", n=_log(rng, 1, 64), graph=graph, lx=lx, ly=ly, lz=lz, wmax=wmax, hmax=hmax,
                    T=rng.randint(3, 32), labels=labels, spp=rng.choice([1, 1, 4]), attempts=_log(rng, 20, 120),
                    icm=labels > 1 and hmax == 0 and rng.random() < 0.75)
    if kind == "gsqa":
        graph = rng.choice(["dimer", "lattice"])
        lx, ly, lz = (rng.randint(3, 9) for _ in range(3))
        n = lx * ly * lz * (2 if graph == "dimer" else 1)
        P, R = rng.randint(8, 80), _log(rng, 8, 1000)
        sweeps = max(5, min(_log(rng, 20, 1000), int(6e9 / (n * P * max(R, 256)))))
        return dict(kind="gsqa", graph=graph, lx=lx, ly=ly, lz=lz, wmax=1, P=P, R=R, sweeps=sweeps)
    if kind == "ladder":
        sweeps = _log(rng, 100, 1500)
        return dict(kind="ladder", n=_log(rng, 1, 64), L=2 * rng.randint(2, 6), chains=rng.randint(8, 40),
                    sweeps=sweeps, tail=max(2, sweeps // 4))
    return dict(kind="mlp", batch=_log(rng, 16, 1024), steps=rng.randint(1, 12))


# ------------------------------------------------------------------ inputs
def _seed(seed, k=0):
    return 1000003 * (int(seed) + 1) + 7919 * k


def _lattice(case, seed, k):
    """(dims, periodic, present or None, J) of instance k; open axes take
    even lengths with vacancies."""
    dims = (case["lx"], case["ly"], case["lz"])
    J = W.ea_couplings(dims, _seed(seed), k)
    if not case["open_xy"]:
        return dims, (1, 1, 1), None, J
    pd, present, Jp = W.pad_odd_open(dims, (0, 0, 1), J)
    return tuple(int(v) for v in pd), (0, 0, 1), present, Jp


def _graph(case, seed, k):
    dims = (case["lx"], case["ly"], case["lz"])
    if case["graph"] == "random":
        return W.sparse_random_graph(case["lx"], 6.0, _seed(seed) % (1 << 40), wmax=case["wmax"], index=k)
    J = W.ea_couplings(dims, _seed(seed), k)
    return W.dimer_embedding(dims, J) if case["graph"] == "dimer" else W.lattice_graph(dims, (1, 1, 1), J)[0]


def _mlp_data(case, seed):
    """Minibatches with the statistics of the ladder network's training set:
    size and coupling features, normalised pilot histograms, and increasing
    32-point ladders from about 0.5 to 3."""
    g = np.random.default_rng(_seed(seed))
    n = case["batch"] * case["steps"]
    X = np.zeros((n, 259), np.float32)
    side = g.choice(np.array([6, 8, 10, 12, 14, 16]), size=n)
    X[:, 0] = side / 16.0
    X[:, 1:3] = 0.5 + g.normal(size=(n, 2)) * (0.3 / side ** 1.5)[:, None]
    centre = np.array([48.0, 36.0, 22.0, 16.0])[None, :] + g.normal(size=(n, 4))
    width = 12.0 / np.sqrt(side)[:, None, None]
    bins = np.arange(64)[None, None, :]
    h = np.round(1024 * np.exp(-0.5 * ((bins - centre[:, :, None]) / width) ** 2))
    X[:, 3:] = (h / h.sum(axis=2, keepdims=True)).reshape(n, 256)
    gaps = (0.04 + 0.05 * np.linspace(0, 1, 31)[None, :] ** 2) * (16.0 / side[:, None]) ** 0.5
    gaps = gaps * (1.0 + 0.2 * g.uniform(-1, 1, size=(n, 31)))
    Y = 0.5 + np.concatenate([np.zeros((n, 1)), np.cumsum(gaps, axis=1)], axis=1)
    return X, Y.astype(np.float32), W.mlp_init(pcomp.MLP_SIZES, int(seed) + 21)


def prepare(case, seed):
    s = dict(case=case)
    kind = case["kind"]
    s["ctx"] = ctx = pcomp.Context(0, _seed(seed) & 0xFFFFFFFF)
    if kind == "sqa":
        s["dims"], s["per"], s["present"], s["J"] = _lattice(case, seed, 0)
        s["gamma"] = W.linear_gamma_schedule(case["sweeps"])
    elif kind == "apt":
        if case["sizes"]:
            rng = np.random.default_rng(case["n"])   # the sizes belong to the case, the couplings to the seed
            side = rng.choice(np.array([int(v) for v in case["sizes"].split(",")]), size=case["n"])
            T = rng.integers(case["T_min"], case["T"] + 1, size=case["n"])
            dims = np.stack([side] * 3, axis=1).astype(np.int32)
            inst = [((int(v),) * 3, None, None, W.ea_couplings((int(v),) * 3, _seed(seed), i))
                    for i, v in enumerate(side)]
        else:
            inst = [_lattice(case, seed, i) for i in range(case["n"])]
            dims = np.array([d for d, _, _, _ in inst], np.int32)
            T = [case["T"]] * case["n"]
        betas = [W.geometric_ladder(int(t)) for t in T]
        J = [j for _, _, _, j in inst]
        if case["open_xy"]:
            pcomp.pc_apt_load_bc(ctx.h, dims, [p for _, p, _, _ in inst], J, betas, case["labels"], 0,
                                 [p for _, _, p, _ in inst])
        else:
            pcomp.pc_apt_load(ctx.h, dims, J, betas, case["labels"], 0)
        s["N"] = [int(np.prod(d)) for d in dims]
    elif kind == "gapt":
        graphs = [_graph(case, seed, i) for i in range(case["n"])]
        h = [W.random_biases(g.n, case["hmax"], _seed(seed, i) % (1 << 40)) for i, g in enumerate(graphs)]
        pcomp.pc_gapt_load(ctx.h, [(g.rp, g.col, g.w) for g in graphs], [W.geometric_ladder(case["T"])] * case["n"],
                           case["labels"], 0, h_list=h if case["hmax"] else None)
        s["N"] = [g.n for g in graphs]
    elif kind == "gsqa":
        s["g"] = _graph(case, seed, 0)
        s["gamma"] = W.linear_gamma_schedule(case["sweeps"])
    elif kind == "ladder":
        L = case["L"]
        s["dims"] = np.tile(np.array([L, L, L], np.int32), (case["n"], 1))
        s["J"] = [W.ea_couplings((L, L, L), _seed(seed), i) for i in range(case["n"])]
    elif kind == "mlp":
        X, Y, params = _mlp_data(case, seed)
        s["stream"] = torch.cuda.Stream()
        pcomp.pc_set_stream(ctx.h, s["stream"].cuda_stream)
        s["net"] = pcomp.Mlp(ctx, params)
        s["net"].set_gap_weight(GAP_WEIGHT)
        s["X"], s["Y"] = torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda()
        s["loss"] = torch.zeros(1, device="cuda")
        torch.cuda.synchronize()
    else:
        raise ValueError(kind)
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    case, h = s["case"], s["ctx"].h
    kind = case["kind"]
    if kind == "sqa":
        N = int(np.prod(s["dims"]))
        if s["present"] is None and not case["spins"]:
            return pcomp.pc_sqa_anneal(h, s["dims"], s["J"], case["P"], SQA_T, s["gamma"], case["R"])
        pcomp.pc_sqa_setup_bc(h, s["dims"], s["per"], s["J"], case["P"], SQA_T, s["gamma"], s["present"])
        return pcomp.pc_sqa_run(h, case["R"], 0, case["P"], N, want_spins=case["spins"])
    if kind == "apt":
        pcomp.pc_apt_run(h, case["attempts"], case["spp"], case["icm"])
        E, hit = pcomp.pc_apt_get_best_all(h, case["n"])
        best = [pcomp.pc_apt_get_best(h, i, n) for i, n in enumerate(s["N"])]
        out = dict(E=E, hit=hit, sweep=np.array([b["sweep"] for b in best]), slot=np.array([b["buf"] for b in best]),
                   spins=np.concatenate([b["spins"] for b in best]))
        if case["state"]:
            out["state"] = [pcomp.pc_apt_get_state(h, i, n, case["T"] * case["labels"])
                            for i, n in enumerate(s["N"])]
        return out
    if kind == "gapt":
        pcomp.pc_gapt_run(h, case["attempts"], case["spp"], case["icm"])
        best = [pcomp.pc_gapt_get_best(h, i, n) for i, n in enumerate(s["N"])]
        return dict(E=np.array([b["E"] for b in best]), sweep=np.array([b["sweep"] for b in best]),
                    slot=np.array([b["buf"] for b in best]), spins=np.concatenate([b["spins"] for b in best]),
                    energies=np.concatenate([pcomp.pc_gapt_get_energies(h, i, case["T"], case["labels"])
                                             for i in range(case["n"])]))
    if kind == "gsqa":
        g = s["g"]
        return pcomp.pc_gsqa_anneal(h, g.rp, g.col, g.w, case["P"], SQA_T, s["gamma"], case["R"])
    if kind == "ladder":
        lad = pcomp.pc_adaptive_ladder(h, s["dims"], s["J"], n_chains=case["chains"], sweeps=case["sweeps"],
                                       tail=case["tail"])
        beta, sigma = np.zeros((case["n"], 64)), np.zeros((case["n"], 64))   # max_len 64, zero beyond a ladder's end
        for i, (b, v, _) in enumerate(lad):
            beta[i, :len(b)], sigma[i, :len(b)] = b, v
        return dict(length=np.array([len(b) for b, _, _ in lad]), beta=beta, sigma=sigma,
                    converged=np.array([c for _, _, c in lad]))
    B = case["batch"]
    for i in range(case["steps"]):
        s["net"].train_step_dev(B, s["X"][i * B:].data_ptr(), s["Y"][i * B:].data_ptr(), 1e-3, s["loss"].data_ptr())
    return dict(params=s["net"].params(), loss=s["loss"])


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    """Bytes: inputs read once, outputs written once.  flops: 32-bit integer
    operations of the spin updates (fp32 operations for the network)."""
    kind = case["kind"]
    if kind == "mlp":
        weights = sum(o * i for i, o in zip(pcomp.MLP_SIZES[:-1], pcomp.MLP_SIZES[1:]))
        return dict(bytes=case["steps"] * (4 * case["batch"] * (259 + 32) + 4 * 6 * weights),
                    flops=case["steps"] * 6 * case["batch"] * weights)
    if kind == "ladder":
        n = case["L"] ** 3
        steps = 20   # ladder steps of a typical instance
        return dict(bytes=case["n"] * (3 * n + 4 * n * case["chains"] / 8 + 16 * steps * case["chains"]),
                    flops=OPS_PER_UPDATE * case["n"] * n * case["chains"] * case["sweeps"] * steps)
    if kind == "apt" and case["sizes"]:
        sides = [int(v) for v in case["sizes"].split(",")]
        n = sum(v ** 3 for v in sides) / len(sides)
    else:
        n = case["lx"] * case["ly"] * case["lz"] * (2 if case.get("graph") == "dimer" else 1)
    if kind in ("sqa", "gsqa"):
        upd = n * case["P"] * case["R"] * case["sweeps"]
        return dict(bytes=3 * n + 8 * case["sweeps"] + 8 * case["R"] * case["P"] +
                    (n * case["P"] * case["R"] if case.get("spins") else 0), flops=OPS_PER_UPDATE * upd)
    reps = case["T"] * case["labels"]
    upd = case["n"] * n * reps * case["attempts"] * case["spp"]
    return dict(bytes=case["n"] * (2 * n * reps / 8 + 3 * n + n + 40), flops=OPS_PER_UPDATE * upd)


# ------------------------------------------------------------------ in 64 bits
def exact(case, seed):
    """The training steps in double precision (plain torch, Adam written out);
    the other kinds return whole numbers, or ladders computed from them by
    billions of random draws."""
    if case["kind"] != "mlp":
        return None
    X, Y, params = _mlp_data(case, seed)
    X, Y = torch.from_numpy(X).double(), torch.from_numpy(Y).double()
    p = [torch.from_numpy(v).double().requires_grad_(True) for Wb in params for v in Wb]
    m, v = [torch.zeros_like(t) for t in p], [torch.zeros_like(t) for t in p]
    B, lr = case["batch"], float(np.float32(1e-3))
    for i in range(case["steps"]):
        x, y = X[i * B:(i + 1) * B], Y[i * B:(i + 1) * B]
        for k in range(4):
            x = x @ p[2 * k].T + p[2 * k + 1]
            if k < 3:
                x = torch.relu(x)
        sp = torch.nn.functional.softplus(x, threshold=1000)
        gap = y[:, 1:] - y[:, :-1]
        loss = ((torch.cumsum(sp, 1) - y) ** 2).mean() + float(np.float32(GAP_WEIGHT)) * (((sp[:, 1:] - gap) / gap) ** 2).mean()
        grads = torch.autograd.grad(loss, p)
        with torch.no_grad():
            for t, g, a, b in zip(p, grads, m, v):
                a.mul_(0.9).add_(g, alpha=0.1)
                b.mul_(0.999).addcmul_(g, g, value=0.001)
                t -= lr * (a / (1 - 0.9 ** (i + 1))) / ((b / (1 - 0.999 ** (i + 1))).sqrt() + 1e-8)
    w = [t.detach().numpy() for t in p]
    return dict(params=[(w[2 * k], w[2 * k + 1]) for k in range(4)], loss=loss.detach().reshape(1))
