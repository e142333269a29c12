"""What this library is measured on: passes that a user's program makes through
the binding, over the sizes, modes and batch shapes it is used at.

Most cases are one time step of a dynamic graph in steady state: a window of
edges that slides over a stream.  The stream has kWindows windows beside a
base graph; a pass inserts the window that comes in and deletes the one that
goes out (dcd_apply_batch or dcd_apply_batch_device), then updates
(dcd_update) and takes the labels, the modularity and the step's counts.  So
every pass changes the graph by the same number of edges, the graph keeps its
size however often the pass is made, and the communities drift from window to
window.  Inputs are drawn on the GPU from the seed alone.

Kinds:
  step      one context: SBM, LFR-style or R-MAT graph; static, base, delta or
            learned mode; batches and labels on the host or on the device
  group     many SBM graphs advanced together (dcd_group)
  train     one epoch of the learned screen's training (dcd_mlp_train)
  quality   modularity of a partition on a device CSR (dcd_modularity_noalloc)
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1904_08553_gb300 import dcd

kWindows = 4
DEV = "cuda"
MODES = {"static": dcd.MODE_STATIC, "base": dcd.MODE_BASE, "delta": dcd.MODE_DELTA, "learned": dcd.MODE_LEARNED}


def listed():
    return [
        # the smallest dynamic graph in use: a small network followed live from a host program
        {"name": "sbm_2k_delta_host", "kind": "step", "graph": "sbm", "n": 2003, "deg": 10.0, "frac": 0.03,
         "mode": "delta", "io": "host", "wmax": 1, "judge": False},
        # the planted-partition configuration: 10,000 vertices, 6,000 edge changes a step, host arrays in and out
        {"name": "sbm_10k_delta_host", "kind": "step", "graph": "sbm", "n": 10_000, "deg": 10.0, "frac": 0.03,
         "mode": "delta", "io": "host", "wmax": 1, "judge": False},
        # a medium social graph (the size the learned screen is trained at), batches made on the GPU
        {"name": "lfr_200k_delta", "kind": "step", "graph": "lfr", "n": 200_003, "deg": 21.0, "frac": 0.03,
         "mode": "delta", "io": "device", "wmax": 1, "judge": False},
        # the benchmark's size and batch: 2M vertices, about 80M directed entries, 6.2M edge changes a step
        {"name": "lfr_2m_delta", "kind": "step", "graph": "lfr", "n": 2_000_000, "deg": 21.0, "frac": 0.074,
         "mode": "delta", "io": "device", "wmax": 1, "judge": False},
        # the same graph at a fine temporal resolution: small batches at a high rate
        {"name": "lfr_2m_delta_fine", "kind": "step", "graph": "lfr", "n": 2_000_000, "deg": 21.0, "frac": 0.0005,
         "mode": "delta", "io": "device", "wmax": 1, "judge": False},
        # the paper's incremental baseline (every vertex re-evaluated from C_{t-1}), host arrays
        {"name": "lfr_1m_base_host", "kind": "step", "graph": "lfr", "n": 1_000_003, "deg": 21.0, "frac": 0.03,
         "mode": "base", "io": "host", "wmax": 1, "judge": False},
        # the paper's static rerun (from singletons at every step): what a first update and a refresh cost
        {"name": "lfr_500k_static", "kind": "step", "graph": "lfr", "n": 500_009, "deg": 21.0, "frac": 0.03,
         "mode": "static", "io": "device", "wmax": 1, "judge": False},
        # the large-scale configuration's generator: skewed degrees, many communities, weights 1..8
        {"name": "rmat_22_delta", "kind": "step", "graph": "rmat", "n": 1 << 22, "deg": 16.0, "frac": 0.0075,
         "mode": "delta", "io": "device", "wmax": 8, "judge": False},
        # the learned screen in service: R_t pruned and widened by the network
        {"name": "lfr_1m_learned", "kind": "step", "graph": "lfr", "n": 1_000_003, "deg": 21.0, "frac": 0.074,
         "mode": "learned", "io": "device", "wmax": 1, "judge": False},
        # the batched form: many uneven graphs, one update for all
        {"name": "group_64_delta", "kind": "group", "G": 64, "nmin": 500, "nmax": 200_000, "frac": 0.02,
         "mode": "delta"},
        # training the screen on collected rows (the benchmark's batch and rate)
        {"name": "train_262k", "kind": "train", "n": 262_144, "batch": 8192, "lr": 2e-3},
        # quality of a partition held by the caller, without device allocation
        {"name": "quality_1m", "kind": "quality", "n": 1_000_000, "deg": 21.0, "wmax": 8},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["step"] * 7 + ["group", "train", "quality"])
    if kind == "group":
        return {"kind": "group", "G": int(_log(rng, 4, 64)), "nmin": rng.randint(100, 2000),
                "nmax": rng.randint(5_000, 200_000), "frac": round(_log(rng, 0.002, 0.05), 5),
                "mode": rng.choice(["delta", "delta", "base"])}
    if kind == "train":
        return {"kind": "train", "n": int(_log(rng, 5_000, 800_000)), "batch": rng.choice([1024, 4096, 8192, 10_000]),
                "lr": 1e-3}
    if kind == "quality":
        return {"kind": "quality", "n": int(_log(rng, 1_000, 1_040_000)), "deg": round(rng.uniform(4, 24), 2),
                "wmax": rng.choice([1, 8])}
    graph = rng.choice(["sbm", "lfr", "lfr", "rmat"])
    mode = rng.choice(["delta", "delta", "delta", "base", "static", "learned"])
    if graph == "sbm":
        n = int(_log(rng, 1_000, 200_000))
    elif graph == "lfr":
        n = int(_log(rng, 20_000, 400_000 if mode == "static" else 1_800_000))
    else:
        n = 1 << rng.randint(12, 18 if mode == "static" else 21)
    return {"kind": "step", "graph": graph, "n": n, "deg": round(rng.uniform(6, 20), 2),
            "frac": round(_log(rng, 0.0005, 0.07), 5), "mode": mode,
            "io": "device" if n > 500_000 else rng.choice(["host", "device"]),
            "wmax": rng.choice([1, 1, 8, 1000] if graph == "rmat" else [1, 1, 8]),
            "judge": mode == "learned" and rng.random() < 0.3}


# ---- inputs --------------------------------------------------------------------

def _rand(m, gen):
    return torch.rand(m, generator=gen, device=DEV, dtype=torch.float64)


def _batch(u, v, w):
    """(k, 3) int32 records without self-loops."""
    keep = u != v
    return torch.stack([u[keep], v[keep], w[keep]], 1).to(torch.int32).contiguous()


def _weights(m, wmax, gen):
    if wmax == 1:
        return torch.ones(m, dtype=torch.int64, device=DEV)
    return torch.randint(1, wmax + 1, (m,), generator=gen, device=DEV)


def _power_law(r, g, lo, hi):
    """Inverse transform of a density x^-g on [lo, hi]."""
    a, b = lo ** (1 - g), hi ** (1 - g)
    return (a + (b - a) * r) ** (1 / (1 - g))


class _Planted:
    """Edge events of a graph with planted communities: an endpoint drawn by
    degree propensity, the other one inside its community (or anywhere, with
    probability mu) by propensity."""

    def __init__(self, graph, n, gen, frac=0.0):
        self.n, self.gen = n, gen
        if graph == "lfr":  # degree exponent 2.5 on [20, 20000], community sizes 1.5 on [100, 50000], mixing 0.3
            self.mu = 0.3
            self.full = _power_law(_rand(n, gen), 2.5, 20.0, float(min(20_000, n / 2)))
            # some vertices (about as many as a window can move, a tenth at most) have few edges in the base graph
            # and a new community in each window, so that every step moves vertices between communities, as drift
            # does in the benchmark's stream
            self.movers = torch.randperm(n, generator=gen, device=DEV)[:int(n * min(0.1, 1.4 * frac))]
            self.prop = self.full.clone()
            self.prop[self.movers] *= 0.02
            sizes = _power_law(_rand(n // 50 + 4, gen), 1.5, 100.0, float(max(200, min(50_000, n // 4)))).long()
        else:  # equal blocks, 80 % of the edges inside
            self.mu = 0.2
            self.prop = self.full = torch.ones(n, dtype=torch.float64, device=DEV)
            self.movers = torch.zeros(0, dtype=torch.int64, device=DEV)
            sizes = torch.full((n // 100 + 2,), 100, dtype=torch.int64, device=DEV)
        ends = torch.cumsum(sizes, 0)
        comm_of_slot = torch.searchsorted(ends, torch.arange(n, device=DEV), right=True)
        self.comm = torch.empty(n, dtype=torch.int64, device=DEV)
        self.comm[torch.randperm(n, generator=gen, device=DEV)] = comm_of_slot
        self._index()

    def _index(self):
        self.order = torch.argsort(self.comm, stable=True)
        cs = torch.cumsum(self.prop[self.order], 0)
        self.cum = cs
        nc = int(self.comm.max()) + 1
        cnt = torch.bincount(self.comm, minlength=nc)
        end = torch.cumsum(cnt, 0)
        zero = torch.zeros(1, dtype=torch.float64, device=DEV)
        tot = torch.cat([zero, cs])
        self.hi = tot[end]
        self.lo = tot[end - cnt]

    def drift(self):
        """The next window: each moving vertex joins the community of a vertex drawn at random."""
        to = torch.randint(0, self.n, (len(self.movers),), generator=self.gen, device=DEV)
        self.comm[self.movers] = self.comm[to].clone()
        self.prop = self.full
        self._index()

    def _pick(self, r):
        return self.order[torch.searchsorted(self.cum, r).clamp_(max=self.n - 1)]

    def events(self, m, wmax):
        out = []
        for m0 in range(0, m, 1 << 24):
            k = min(1 << 24, m - m0)
            u = self._pick(_rand(k, self.gen) * self.cum[-1])
            c = self.comm[u]
            r, any_ = _rand(k, self.gen), _rand(k, self.gen) < self.mu
            v = self._pick(torch.where(any_, r * self.cum[-1], self.lo[c] + r * (self.hi[c] - self.lo[c])))
            out.append(_batch(u, v, _weights(k, wmax, self.gen)))
        return torch.cat(out) if out else torch.zeros((0, 3), dtype=torch.int32, device=DEV)


class _Rmat:
    """R-MAT (0.57, 0.19, 0.19, 0.05) over 2^s vertices with permuted ids."""

    def __init__(self, n, gen):
        self.n, self.gen = n, gen
        self.scale = n.bit_length() - 1
        self.perm = torch.randperm(n, generator=gen, device=DEV)

    def drift(self):
        pass

    def events(self, m, wmax):
        out = []
        for m0 in range(0, m, 1 << 24):
            k = min(1 << 24, m - m0)
            u = torch.zeros(k, dtype=torch.int64, device=DEV)
            v = torch.zeros(k, dtype=torch.int64, device=DEV)
            for _ in range(self.scale):
                r = torch.rand(k, generator=self.gen, device=DEV)
                u = 2 * u + (r >= 0.76)
                v = 2 * v + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
            out.append(_batch(self.perm[u], self.perm[v], _weights(k, wmax, self.gen)))
        return torch.cat(out) if out else torch.zeros((0, 3), dtype=torch.int32, device=DEV)


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _screen(seed):
    """The parameters of a screen network: the score rises as the weight to the
    best other community comes near the weight to the own one (what training
    finds), spread over all hidden units."""
    r = np.random.default_rng(seed)
    W1 = 0.02 * r.standard_normal((12, 64))
    W1[6] += 1.0
    W1[5] -= 1.0
    W2 = np.eye(64) + 0.01 * r.standard_normal((64, 64))
    w3 = np.full(64, 16 / 64)
    return np.concatenate([W1.ravel(), np.ones(64), W2.ravel(), np.zeros(64), w3, [-14.4]]).astype(np.float32)


def _prepare_step(c, seed):
    gen = _gen(seed)
    n, total = c["n"], int(c["n"] * c["deg"])
    k = max(1, int(total * c["frac"]))
    src = _Rmat(n, gen) if c["graph"] == "rmat" else _Planted(c["graph"], n, gen, c["frac"])
    parts = [src.events(total - kWindows * k, c["wmax"])]
    for _ in range(kWindows):
        src.drift()
        parts.append(src.events(k, c["wmax"]))
    load = torch.cat([parts[0]] + parts[2:])  # all but the first window
    s = {"case": c, "step": 0}
    s["ctx"] = ctx = dcd.Context(n, mode=MODES[c["mode"]])
    ctx.reserve(2 * total, total)
    torch.cuda.synchronize()
    ctx.apply_batch_device(load, len(load), None, 0)
    ctx.update(labels_out=None)
    if c["mode"] == "learned":
        s["mlp"] = dcd.Mlp(seed=seed)
        s["mlp"].params = _screen(seed)
        ctx.set_screen(s["mlp"], theta_keep=0.3, theta_add=0.9, judge=c["judge"])
    win = parts[1:]
    if c["io"] == "host":
        win = [w.cpu().numpy() for w in win]
        s["labels"] = "host"
    else:
        s["labels"] = torch.empty(n, dtype=torch.int32, device=DEV)
    s["win"] = win
    return s


def _counts(st):
    return [int(x) for x in (st.r_size, st.levels, st.iters_total, st.moves_total, st.communities, st.nnz, st.m2)]


def _run_step(s):
    ctx, k = s["ctx"], s["step"]
    ins, out = s["win"][k % kWindows], s["win"][(k + 1) % kWindows]
    if s["case"]["io"] == "host":
        ctx.apply_batch(ins, out)
    else:
        ctx.apply_batch_device(ins, len(ins), out, len(out))
    labels, q, st = ctx.update(labels_out=s["labels"])
    s["step"] = k + 1
    return {"labels": labels, "q": float(q), "counts": np.array(_counts(st), np.int64)}


def _group_sizes(c):
    r = np.random.default_rng(c["G"] * 7 + c["nmax"])
    n = np.exp(r.uniform(np.log(c["nmin"]), np.log(c["nmax"]), c["G"])).astype(np.int64)
    return n, r.uniform(8, 32, c["G"])


def _prepare_group(c, seed):
    gen = _gen(seed)
    sizes, deg = _group_sizes(c)
    grp = dcd.Group(sizes, mode=MODES[c["mode"]])
    win = [[] for _ in range(kWindows)]
    for g in range(c["G"]):
        n = int(sizes[g])
        total = int(n * deg[g] / 2)
        k = max(1, int(total * c["frac"]))
        e = _Planted("sbm", n, gen).events(total, 1).cpu().numpy()
        grp.apply_batch(g, e[k:])
        for i in range(kWindows):
            win[i].append(np.ascontiguousarray(e[i * k:(i + 1) * k]))
    grp.update(labels_out=None)
    return {"case": c, "grp": grp, "win": win, "step": 0}


def _run_group(s):
    grp, k = s["grp"], s["step"]
    ins, out = s["win"][k % kWindows], s["win"][(k + 1) % kWindows]
    for g in range(grp.G):
        grp.apply_batch(g, ins[g], out[g])
    labels, q, st = grp.update()
    s["step"] = k + 1
    return {"labels": labels, "q": q, "counts": np.array([_counts(x) for x in st], np.int64)}


def _train_rows(c, seed):
    """Rows with the ranges of the screen's features, and move labels that
    follow the two community shares with noise; 5 % of the rows move."""
    gen = _gen(seed)
    n = c["n"]
    r = torch.rand((n, 16), generator=gen, device=DEV)
    deg = _power_law(r[:, 0], 2.5, 8.0, 20_000.0)
    eC = r[:, 1] ** 0.5
    eB = (1 - eC) * r[:, 2]
    X = torch.stack([torch.log1p(deg), torch.log1p(deg * (1 + r[:, 3])), torch.log1p(8 * r[:, 4] ** 4),
                     torch.log1p(2 * r[:, 5] ** 8), r[:, 6] ** 6, eC, eB, eB - eC, 0.01 * r[:, 7], 0.01 * r[:, 8],
                     torch.log1p(5000 * r[:, 9]), (r[:, 10] < 0.9).float()], 1).contiguous()
    y = ((eB - eC + 0.2 * (r[:, 11] - 0.5)) > 0.25).float().contiguous()
    return X, y


def _train_params(c, seed):
    r = np.random.default_rng(seed)
    W1, W2 = r.uniform(-0.7, 0.7, 768), r.uniform(-0.3, 0.3, 4096)
    return np.concatenate([W1, np.zeros(64), W2, np.zeros(64), r.uniform(-0.3, 0.3, 64), [0.0]]).astype(np.float32)


def _prepare_train(c, seed):
    X, y = _train_rows(c, seed)
    m = dcd.Mlp(seed=seed)
    m.params = _train_params(c, seed)
    torch.cuda.synchronize()
    return {"case": c, "mlp": m, "X": X, "y": y}


def _run_train(s):
    c, m = s["case"], s["mlp"]
    loss = m.train(s["X"], s["y"], c["n"], batch=c["batch"], epochs=1, lr=c["lr"])
    return {"params": m.params, "loss": loss}


def _exact_train(c, seed):
    """The epoch in 64 bits: mini-batches in row order, mean cross-entropy, Adam."""
    X, y = _train_rows(c, seed)
    X, y = X.double(), y.double()
    P = torch.from_numpy(_train_params(c, seed)).double().to(DEV).requires_grad_(True)
    m, v = torch.zeros_like(P), torch.zeros_like(P)
    loss = None
    for t, r in enumerate(range(0, c["n"], c["batch"]), 1):
        x, t_y = X[r:r + c["batch"]], y[r:r + c["batch"]]
        h = torch.relu(x @ P[:768].view(12, 64) + P[768:832])
        h = torch.relu(h @ P[832:4928].view(64, 64) + P[4928:4992])
        loss = torch.nn.functional.binary_cross_entropy_with_logits(h @ P[4992:5056] + P[5056], t_y)
        g, = torch.autograd.grad(loss, P)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        with torch.no_grad():
            P -= c["lr"] * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
    return {"params": P.detach().cpu().numpy(), "loss": float(loss)}


def _quality_graph(c, seed):
    gen = _gen(seed)
    n = c["n"]
    src = _Planted("lfr", n, gen)
    e = src.events(int(n * c["deg"]), c["wmax"]).long()
    lo, hi = torch.minimum(e[:, 0], e[:, 1]), torch.maximum(e[:, 0], e[:, 1])
    key, inv = torch.unique(lo * n + hi, return_inverse=True)
    w = torch.zeros(len(key), dtype=torch.int64, device=DEV).index_add_(0, inv, e[:, 2])
    u, v = torch.cat([key // n, key % n]), torch.cat([key % n, key // n])
    order = torch.argsort(u * n + v)
    u, col, w = u[order], v[order].to(torch.int32), torch.cat([w, w])[order].to(torch.int32)
    rp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rp[1:] = torch.cumsum(torch.bincount(u, minlength=n), 0)
    return rp, col.contiguous(), w.contiguous(), src.comm.to(torch.int32).contiguous()


def _prepare_quality(c, seed):
    rp, col, w, lab = _quality_graph(c, seed)
    torch.cuda.synchronize()
    return {"case": c, "rp": rp, "col": col, "w": w, "lab": lab}


def _run_quality(s):
    q, m2 = dcd.dcd_modularity_noalloc(s["case"]["n"], s["rp"], s["col"], s["w"], s["lab"])
    return {"q": q, "m2": m2}


def _exact_quality(c, seed):
    rp, col, w, lab = _quality_graph(c, seed)
    n = c["n"]
    src = torch.repeat_interleave(torch.arange(n, device=DEV), rp[1:] - rp[:-1])
    wl = w.long()
    a = torch.zeros(n, dtype=torch.int64, device=DEV).index_add_(0, lab[src].long(), wl).cpu().numpy()
    m2 = int(wl.sum())
    inside = int(wl[lab[src] == lab[col.long()]].sum())
    sq = sum(int(x) * int(x) for x in a[a > 0])
    return {"q": (m2 * inside - sq) / (m2 * m2), "m2": None}


# ---- the interface ---------------------------------------------------------------

def prepare(case, seed):
    return {"step": _prepare_step, "group": _prepare_group, "train": _prepare_train,
            "quality": _prepare_quality}[case["kind"]](case, seed)


def run(state):
    return {"step": _run_step, "group": _run_group, "train": _run_train,
            "quality": _run_quality}[state["case"]["kind"]](state)


def exact(case, seed):
    """Labels and counts are whole numbers and a step's modularity follows from
    them, so only the network and the partition's quality have a value in 64 bits."""
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case["kind"] == "quality":
        return _exact_quality(case, seed)
    return None


def work(case):
    """The graph read once (8 bytes a directed entry), the batch read and the
    changed entries written, the labels read and written; one multiply-add a
    directed entry.  Training: forward, two backward products."""
    k = case["kind"]
    if k == "train":
        f = 12 * 64 + 64 * 64 + 64
        return {"bytes": case["n"] * 13 * 4 + 2 * 5057 * 4, "flops": case["n"] * (6 * f - 2 * 12 * 64)}
    if k == "quality":
        nnz = 2 * case["n"] * case["deg"]
        return {"bytes": 8 * nnz + 12 * case["n"], "flops": 2 * nnz}
    if k == "group":
        sizes, deg = _group_sizes(case)
        n, edges = int(sizes.sum()), float((sizes * deg / 2).sum())
    else:
        n, edges = case["n"], case["n"] * case["deg"]
    changed = 2 * edges * case["frac"]
    return {"bytes": 8 * 2 * edges + changed * (12 + 2 * 8) + 8 * n, "flops": 2 * 2 * edges}
