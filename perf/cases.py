"""Workloads of the library, each one pass through its public entry points.

A case is a dict of plain values; its "kind" says what a pass does:

* "train":  minibatch or Hogwild training of one or both orders, then the
            trained tables read into the caller's device buffers;
* "alias":  both alias tables of a new graph, read into the caller's buffers;
* "warm":   the warm start of arriving nodes: MLP creation, the inputs of a
            sample of known nodes, the Adam steps, then the inputs and the
            predictions of the new nodes;
* "eval":   link-prediction AUC of held-out edges against non-edges, and the
            LINE loss.

Graphs are R-MAT (0.57, 0.19, 0.19, 0.05; edge factor 16; symmetrised;
duplicates merged into integer weights) or directed Chung-Lu (power-law
out-degrees of exponent 2.2, lognormal(0,1) weights), generated on the GPU.
Tables start from a checkpoint-like state: every row's values have a share
that grows with the log of the node's degree, as trained rows do.

``exact`` restates each pass in 64-bit torch arithmetic, sampling included.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2604_09419_gb300 import line as L

DEV = "cuda"
LR0, FLOOR = 0.025, 1e-4


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def _train(name, graph, nodes, orders, dim, K, batch, samples, dtype="f32", mode="batched", walk=0, window=0, lam=0.0,
           alpha_neg=1.0, fresh=False):
    return {"name": name, "kind": "train", "graph": graph, "nodes": nodes, "orders": orders, "dim": dim, "K": K,
            "batch": batch, "samples": samples, "dtype": dtype, "mode": mode, "walk": walk, "window": window,
            "lam": lam, "alpha_neg": alpha_neg, "fresh": fresh}


def listed():
    return [
        # a whole run on a small graph (1,000 nodes, d = 16, minibatch 256,
        # 100,000 samples, fresh tables): launches and latency only
        _train("tiny_whole_run", "dchung", 1000, "2", 16, 5, 256, 100_000, fresh=True),
        # first-order training with the paper's K = 1 on a mid-size graph, an
        # odd batch, a ragged last batch, weight decay and alpha_neg in use
        _train("rmat14_o1_d64_k1_ragged", "rmat", 1 << 14, "1", 64, 1, 1000, 300_001, lam=1e-3, alpha_neg=0.5),
        # wide rows and many negatives
        _train("rmat18_o2_d256_k10", "rmat", 1 << 18, "2", 256, 10, 2048, 1 << 19),
        # the benchmark workload: both orders on R-MAT 20, FP32, B = 4096;
        # 2^22 samples between two looks at the tables
        _train("rmat20_orders_f32", "rmat", 1 << 20, "12", 128, 5, 4096, 1 << 22),
        # one order alone in BF16, as the phase before new nodes arrive runs
        _train("rmat20_o2_bf16", "rmat", 1 << 20, "2", 128, 5, 4096, 1 << 22, dtype="bf16"),
        # the largest: both orders in BF16, tables and graph far beyond L2
        _train("rmat22_orders_bf16", "rmat", 1 << 22, "12", 128, 5, 4096, 1 << 23, dtype="bf16"),
        # weighted directed graph with the batch the autotuner takes there
        _train("dchung22_o2_bf16_b16384", "dchung", 1 << 22, "2", 128, 5, 16384, 1 << 23, dtype="bf16"),
        # positive pairs from random walks (length 100, window 2), both orders
        _train("rmat20_walk_orders", "rmat", 1 << 20, "12", 128, 5, 4096, 1 << 22, walk=100, window=2),
        # the per-pair lock-free schedule
        _train("rmat20_hogwild_o2", "rmat", 1 << 20, "2", 128, 5, 4096, 1 << 22, mode="hogwild"),
        # a graph arrives: both alias tables (31M arcs, integer weights)
        {"name": "alias_rmat20", "kind": "alias", "graph": "rmat", "nodes": 1 << 20},
        # nodes arrive: the MLP's fit on 65,536 known nodes (16 Adam steps of
        # 16,384) and the new nodes' rows (10% of the nodes)
        {"name": "warm_rmat20", "kind": "warm", "graph": "rmat", "nodes": 1 << 20, "dim": 128, "dtype": "bf16",
         "act": "bf16", "hidden": 256, "sample": 1 << 16, "batch": 16384, "steps": 16},
        # a look at the quality: 10% held-out edges against as many non-edges,
        # and the loss over 2^20 samples, both orders' tables
        {"name": "eval_rmat20", "kind": "eval", "graph": "rmat", "nodes": 1 << 20, "dim": 128, "dtype": "f32",
         "score": "dot", "m": 1 << 20, "K": 5},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_graph(rng, top):
    """An R-MAT graph (a power of two nodes) or a directed one of any size."""
    if rng.random() < 0.7:
        return "rmat", 1 << rng.randint(12, top)
    return "dchung", _log_int(rng, 1000, 1 << top)


def draw(rng):
    r = rng.random()
    if r < 0.64:
        graph, nodes = _draw_graph(rng, 22)
        mode, walk, window = "batched", 0, 0
        q = rng.random()
        if q < 0.15:
            mode = "hogwild"
        elif q < 0.3 and graph == "rmat":
            walk = rng.randint(20, 100)
            window = rng.randint(1, 5)
        dim = rng.choice([16, 32, 64, 128, 128, 128, 256])
        if dim == 256 and nodes > 1 << 20:
            nodes = 1 << 20
        K = rng.choice([1, 2, 3, 5, 5, 5, 6, 8, 10])
        orders = rng.choice(["1", "2", "2", "12"])
        batch = _log_int(rng, 200, 16384) if rng.random() < 0.6 else rng.choice([1024, 4096, 4096, 8192])
        # at most the row traffic of the listed benchmark workload, and at
        # most 2,000 batches
        rows = (2 if orders == "12" else 1) * (K + 2) * dim
        most = min((1 << 22) * 2 * 7 * 128 // rows, 2000 * batch, 1 << 22)
        samples = _log_int(rng, min(most // 2, 40_000), most)
        case = _train("", graph, nodes, orders, dim, K, batch, samples, dtype=rng.choice(["f32", "f32", "bf16"]),
                      mode=mode, walk=walk, window=window, lam=rng.choice([0.0, 0.0, 1e-3]),
                      alpha_neg=rng.choice([1.0, 1.0, 0.5]), fresh=rng.random() < 0.2)
        del case["name"]
        return case
    if r < 0.76:
        graph, nodes = _draw_graph(rng, 21)
        return {"kind": "alias", "graph": graph, "nodes": nodes}
    if r < 0.9:
        act = rng.choice(["bf16", "bf16", "bf16", "f32"])
        nodes = 1 << rng.randint(14, 20)
        batch = _log_int(rng, 500, 16384 if act == "bf16" else 4096)
        return {"kind": "warm", "graph": "rmat", "nodes": nodes, "dim": rng.choice([64, 128, 128]),
                "dtype": rng.choice(["bf16", "f32"]), "act": act, "hidden": rng.choice([128, 256, 256]),
                "sample": _log_int(rng, 2000, min(1 << 16, nodes // 4)), "batch": batch, "steps": rng.randint(4, 16)}
    graph, nodes = _draw_graph(rng, 20)
    return {"kind": "eval", "graph": graph, "nodes": nodes, "dim": rng.choice([32, 64, 128, 128]),
            "dtype": rng.choice(["bf16", "f32"]), "score": rng.choice(["dot", "dot", "cosine"]),
            "m": _log_int(rng, 20_000, 1 << 20), "K": rng.choice([1, 5, 5, 10])}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _generator(seed, stream):
    return torch.Generator(device=DEV).manual_seed(seed * 1000 + stream)


def _make_graph(case, seed):
    """(src, dst, w) of the case's graph: int32, int32, float32 arcs sorted by (src, dst)."""
    n = case["nodes"]
    g = _generator(seed, 1)
    if case["graph"] == "rmat":
        m = 16 * n
        src = torch.zeros(m, dtype=torch.int64, device=DEV)
        dst = torch.zeros(m, dtype=torch.int64, device=DEV)
        for _ in range(n.bit_length() - 1):
            u = torch.rand(m, generator=g, device=DEV)
            src = 2 * src + (u >= 0.76)
            dst = 2 * dst + (((u >= 0.57) & (u < 0.76)) | (u >= 0.95))
        keep = src != dst
        src, dst = src[keep], dst[keep]
        key, count = torch.unique(torch.cat([src * n + dst, dst * n + src]), return_counts=True)
        w = count.to(torch.float32)
    else:
        m = 16 * n
        # summed on the host: the GPU's running sum differs from run to run
        cdf = np.cumsum(np.arange(1, n + 1, dtype=np.float64) ** (-1.0 / 1.2))
        cdf = torch.from_numpy(cdf / cdf[-1]).to(DEV)
        src = torch.searchsorted(cdf, torch.rand(m, generator=g, device=DEV, dtype=torch.float64)).clamp_(max=n - 1)
        dst = torch.randint(0, n, (m,), generator=g, device=DEV)
        w = torch.exp(torch.randn(m, generator=g, device=DEV))
        keep = src != dst
        key, order = torch.sort((src * n + dst)[keep], stable=True)
        first = torch.ones_like(key, dtype=torch.bool)
        first[1:] = key[1:] != key[:-1]
        key, w = key[first], w[keep][order][first]
    return (key // n).to(torch.int32), (key % n).to(torch.int32), w.contiguous()


def _make_table(n, dim, logdeg, dtype, seed, stream):
    g = _generator(seed, stream)
    t = torch.randn(n, dim, generator=g, device=DEV) + 0.15 * logdeg[:, None] * torch.randn(dim, generator=g, device=DEV)
    t *= dim ** -0.5
    return t.to(torch.bfloat16) if dtype == "bf16" else t


def _log_degree(n, src):
    return torch.log1p(torch.bincount(src.long(), minlength=n).to(torch.float32))


def _split_edges(n, src, dst, w, seed):
    """1.5 n undirected edges (about 10% on R-MAT) held out: (kept arcs, held src, held dst)."""
    once = torch.nonzero(src < dst).flatten()
    pick = once[torch.randperm(once.numel(), generator=_generator(seed, 4), device=DEV)[: n + n // 2]]
    hs, hd = src[pick].contiguous(), dst[pick].contiguous()
    key = torch.minimum(src, dst).long() * n + torch.maximum(src, dst)
    held = torch.isin(key, hs.long() * n + hd)
    return src[~held], dst[~held], w[~held], hs, hd


def _non_edges(n, src, dst, count, seed):
    arcs = src.long() * n + dst.long()
    g = _generator(seed, 5)
    got = torch.empty(0, dtype=torch.int64, device=DEV)
    while got.numel() < count:
        key = torch.randint(0, n * n, (2 * count + 1024,), generator=g, device=DEV)
        at = torch.searchsorted(arcs, key).clamp_(max=arcs.numel() - 1)
        got = torch.cat([got, key[(arcs[at] != key) & (key // n != key % n)]])
    got = got[:count]
    return (got // n).to(torch.int32), (got % n).to(torch.int32)


def _warm_inputs(case, seed):
    n = case["nodes"]
    src, dst, w = _make_graph(case, seed)
    table = _make_table(n, case["dim"], _log_degree(n, src), case["dtype"], seed, 2)
    g = _generator(seed, 6)
    order = torch.randperm(n, generator=g, device=DEV)
    new, ids = torch.sort(order[: n // 10])[0].to(torch.int32), order[n // 10:]
    known = torch.ones(n, dtype=torch.bool, device=DEV)
    known[new.long()] = False
    sample = ids[torch.randint(0, ids.numel(), (case["sample"],), generator=g, device=DEV)].to(torch.int32)
    return src, dst, w, table, known.to(torch.uint8), new, sample


def _train_tables(case, seed, src):
    """{(order, which): table} of a resumed run."""
    n, logdeg = case["nodes"], _log_degree(case["nodes"], src)
    got = {}
    for o in case["orders"]:
        for which in (L.WHICH_U, L.WHICH_C)[: int(o)]:
            got[int(o), which] = _make_table(n, case["dim"], logdeg, case["dtype"], seed, 10 * int(o) + which)
    return got


def _code(dtype):
    return L.DTYPE_BF16 if dtype == "bf16" else L.DTYPE_F32


def _context():
    return L.Context(0, torch.cuda.current_stream().cuda_stream)


def prepare(case, seed):
    n = case["nodes"]
    if case["kind"] == "train":
        src, dst, w = _make_graph(case, seed)
        ctx = _context()
        ctx.build_alias(n, src, dst, w)
        out = {}
        for (o, which), t in _train_tables(case, seed, src).items():
            if which == L.WHICH_U:
                ctx.init_embeddings(o, case["dim"], _code(case["dtype"]), seed + 1)
            if not case["fresh"]:
                ctx.set_embeddings(o, which, t, _code(case["dtype"]))
            out[o, which] = torch.empty_like(t)
        opts = L.train_opts_default()
        opts.batch, opts.lambda_, opts.alpha_neg = case["batch"], case["lam"], case["alpha_neg"]
        opts.mode = L.MODE_HOGWILD if case["mode"] == "hogwild" else L.MODE_BATCHED
        opts.walk_length, opts.window = case["walk"], case["window"]
        return {"case": case, "seed": seed, "ctx": ctx, "opts": opts, "out": out, "total": 20 * int(src.numel()), "offset": 0}
    if case["kind"] == "alias":
        src, dst, w = _make_graph(case, seed)
        # buffers for any graph of this size (at most 32 n arcs)
        out = [torch.zeros(k, dtype=torch.int32, device=DEV) for k in (32 * n, 32 * n, n, n)]
        return {"case": case, "ctx": _context(), "graph": (src, dst, w), "out": out}
    if case["kind"] == "warm":
        src, dst, w, table, known, new, sample = _warm_inputs(case, seed)
        ctx = _context()
        ctx.build_alias(n, src, dst, w)
        ctx.init_embeddings(2, case["dim"], _code(case["dtype"]), seed + 1)
        ctx.set_embeddings(2, L.WHICH_U, table, _code(case["dtype"]))
        y = torch.empty(new.numel(), case["dim"], device=DEV)
        return {"case": case, "seed": seed, "ctx": ctx, "known": known, "new": new, "sample": sample, "y": y}
    ksrc, kdst, kw, ps, pd, ns, nd, tables = _eval_inputs(case, seed)
    ctx = _context()
    ctx.build_alias(n, ksrc, kdst, kw)
    for (o, which), t in tables.items():
        if which == L.WHICH_U:
            ctx.init_embeddings(o, case["dim"], _code(case["dtype"]), seed + 1)
        ctx.set_embeddings(o, which, t, _code(case["dtype"]))
    scores = torch.empty(ps.numel() + ns.numel(), device=DEV)
    return {"case": case, "seed": seed, "ctx": ctx, "pairs": (ps, pd, ns, nd), "scores": scores}


def _eval_inputs(case, seed):
    n = case["nodes"]
    src, dst, w = _make_graph(case, seed)
    ksrc, kdst, kw, ps, pd = _split_edges(n, src, dst, w, seed)
    ns, nd = _non_edges(n, src, dst, ps.numel(), seed)
    return ksrc, kdst, kw, ps, pd, ns, nd, _train_tables({**case, "orders": "12"}, seed, src)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    case, ctx = state["case"], state["ctx"]
    if case["kind"] == "train":
        dim, K, seed = case["dim"], case["K"], state["seed"] + 7
        if case["fresh"]:
            for o in case["orders"]:
                ctx.init_embeddings(int(o), dim, _code(case["dtype"]), state["seed"] + 1)
        opts = state["opts"]
        opts.sample_offset = state["offset"]
        lr = {"lr0": LR0, "schedule": 1, "floor_frac": FLOOR, "total": state["total"]}
        if case["orders"] == "12":
            ctx.train_orders(dim, K, case["samples"], seed, opts=opts, **lr)
        else:
            ctx.train_steps(int(case["orders"]), dim, K, case["samples"], seed, opts=opts, **lr)
        if not case["fresh"]:
            # the next pass goes on from here, at a batch boundary
            state["offset"] += -(-case["samples"] // case["batch"]) * case["batch"]
        for (o, which), t in state["out"].items():
            ctx.get_embeddings(o, which, t, _code(case["dtype"]))
        return [t for _, t in sorted(state["out"].items())]
    if case["kind"] == "alias":
        src, dst, w = state["graph"]
        ctx.build_alias(case["nodes"], src, dst, w)
        out = state["out"]
        ctx.get_alias(L.TABLE_EDGE, out[0], out[1])
        ctx.get_alias(L.TABLE_NEG, out[2], out[3])
        return out
    if case["kind"] == "warm":
        ctx.mlp_create(2, hidden=case["hidden"], act_dtype=_code(case["act"]), seed=state["seed"] + 9)
        ctx.mlp_features_rows(state["known"], state["sample"])
        losses = ctx.mlp_train(state["sample"], steps=case["steps"], batch=case["batch"], lr=1e-3, seed=state["seed"] + 10)
        ctx.mlp_features_rows(state["known"], state["new"])
        ctx.mlp_predict(state["new"], state["y"])
        return {"losses": losses.tolist(), "params": ctx.mlp_get_params(), "y": state["y"]}
    score = L.SCORE_COSINE if case["score"] == "cosine" else L.SCORE_DOT
    auc, counts = ctx.eval_auc(3, *state["pairs"], scores=state["scores"], score=score)
    loss = ctx.eval_loss(2, case["K"], state["seed"] + 3, case["m"])
    return {"scores": state["scores"], "auc": auc, "counts": list(counts), "loss": loss}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    n = case["nodes"]
    arcs = 30 * n if case["graph"] == "rmat" else 16 * n
    es = lambda t: 2 if t == "bf16" else 4  # noqa: E731
    if case["kind"] == "train":
        # per update: its K + 2 rows read and written, its 8-byte alias
        # entries and its arc's ends; the tables copied out once
        k = len(case["orders"])
        tables = sum(int(o) for o in case["orders"]) * n * case["dim"] * es(case["dtype"])
        per = 2 * (case["K"] + 2) * case["dim"] * es(case["dtype"]) + 8 * (case["K"] + 1) + 8
        return {"bytes": k * case["samples"] * per + 2 * tables, "flops": k * case["samples"] * (case["K"] + 1) * case["dim"] * 6}
    if case["kind"] == "alias":
        # arcs in (12 bytes each), both tables out (8 bytes an entry)
        return {"bytes": 12 * arcs + 8 * arcs + 8 * n, "flops": 4 * (arcs + n)}
    if case["kind"] == "warm":
        d, H = case["dim"], case["hidden"]
        P = (d + 1 + 15) // 16 * 16
        row = d * es(case["dtype"])
        # inputs: every arc of the requested nodes (its head, the known mark
        # and the neighbour's row); a step: its rows' inputs and targets; the
        # parameters and their two moments read and written
        deg = arcs / n
        params = 4 * (H * P + H + d * H + d)
        seen = case["sample"] + 0.1 * n
        per_step = case["batch"] * (P * es(case["act"]) + row) + 6 * params
        return {"bytes": int(seen * deg * (5 + row) + case["steps"] * per_step + 0.1 * n * 4 * d),
                "flops": int(6 * case["steps"] * case["batch"] * H * (P + d) + 0.2 * n * H * (P + d))}
    pairs = 0.1 * arcs  # held-out edges (half the held arcs) and as many non-edges
    row = case["dim"] * es(case["dtype"])
    return {"bytes": int(pairs * (2 * 2 * row + 12) + case["m"] * (case["K"] + 2) * row),
            "flops": int(pairs * 4 * case["dim"] + case["m"] * (case["K"] + 1) * case["dim"] * 2)}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
_M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Words of Philox4x32-10 at counter (c0, c1, c2, c3), int64 tensors of 32-bit values."""
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
        a, b = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((b >> 32) & _M32) ^ c1 ^ k0, b & _M32, ((a >> 32) & _M32) ^ c3 ^ k1, a & _M32
    return c0, c1, c2, c3


def _words(seed, domain, t, call):
    z = torch.zeros_like(t)
    return _philox(t & _M32, (t >> 32) & _M32, z + call, z + domain, seed)


def _mulhi(w, n):
    return (w[1] * n + (((w[0] * n) >> 32) & _M32)) >> 32


def _tree_sum(x):
    while x.numel() > 1:
        x = torch.nn.functional.pad(x, (0, -x.numel() % 1024)).view(-1, 1024).clone()
        s = 512
        while s:
            x[:, :s] += x[:, s:2 * s].clone()
            s //= 2
        x = x[:, 0].contiguous()
    return x


def _alias(x):
    """(thr, alias) of weights x: floor masses, the remainder spread, sweep pairing."""
    n, Q = x.numel(), 1 << 32
    m = torch.floor(x * (n * float(Q) / _tree_sum(x))).to(torch.int64)
    D = n * Q - int(m.sum())
    on = x > 0 if D > 0 else m >= 1
    rank = torch.cumsum(on, 0) - 1
    if D > 0:
        q, r = divmod(D, int(on.sum()))
        m += on * (q + (rank < r))
    else:
        m -= (on & (rank < -D)).long()
    thr = torch.full((n,), _M32, dtype=torch.int64, device=DEV)
    alias = torch.arange(n, device=DEV)
    li, hi = torch.nonzero(m < Q).flatten(), torch.nonzero(m > Q).flatten()
    if li.numel():
        dp, ep = torch.cumsum(Q - m[li], 0), torch.cumsum(m[hi] - Q, 0)
        thr[li] = m[li]
        alias[li] = hi[torch.searchsorted(ep, dp - (Q - m[li]))]
        j = torch.searchsorted(dp, ep[:-1], right=True)
        thr[hi[:-1]] = Q - (dp[j] - ep[:-1])
        alias[hi[:-1]] = hi[1:]
    return thr, alias


class _Sampler:
    def __init__(self, n, src, dst, w):
        self.n, self.m, self.src, self.dst = n, src.numel(), src.long(), dst.long()
        w = w.double()
        self.first = torch.searchsorted(self.src, torch.arange(n + 1, device=DEV))
        self.deg = torch.zeros(n, dtype=torch.float64, device=DEV).index_add_(0, self.src, w)
        # running weights over all arcs, for the walks (integer weights: exact)
        self.cum = torch.cumsum(w, 0)
        self.base = torch.cat([torch.zeros(1, dtype=torch.float64, device=DEV), self.cum])[self.first[:-1]]
        self.edge = _alias(w)
        self.neg = _alias(torch.sqrt(self.deg) * torch.sqrt(torch.sqrt(self.deg)))

    def pick(self, table, n, w):
        i = _mulhi(w, n)
        return torch.where(w[2] < table[0][i], i, table[1][i])

    def records(self, seed, domain, t, K):
        e = self.pick(self.edge, self.m, _words(seed, domain, t, 0))
        cols = [self.src[e], self.dst[e]]
        cols += [self.pick(self.neg, self.n, _words(seed, domain, t, j)) for j in range(1, K + 1)]
        return torch.stack(cols, 1)

    def walk_pairs(self, seed, t, Lw, W):
        """(u, v) of samples t: pairs of the walks (integer arc weights)."""
        P = Lw * W - W * (W - 1) // 2
        w0 = int(t[0]) // P
        wk = torch.arange(w0, int(t[-1]) // P + 1, device=DEV)
        e = self.pick(self.edge, self.m, _words(seed, 8, wk, 0))
        nodes = [self.src[e], self.dst[e]]
        for i in range(1, Lw):
            x = nodes[-1]
            w = _words(seed, 8, wk, i)
            u = ((w[1] << 21) | (w[0] >> 11)).double() * 2.0 ** -53
            at = torch.searchsorted(self.cum, self.base[x] + torch.floor(u * self.deg[x]) + 1)
            at = torch.minimum(at, self.first[x + 1] - 1)
            nodes.append(torch.where(self.deg[x] > 0, self.dst[at.clamp(min=0)], nodes[-2]))
        nodes = torch.stack(nodes, 1)
        ij = torch.tensor([(i, i + k) for i in range(Lw) for k in range(1, W + 1) if i + k <= Lw], device=DEV)
        row, pair = t // P - w0, ij[t % P]
        return nodes[row, pair[:, 0]], nodes[row, pair[:, 1]]


def _fresh_table(n, dim, seed):
    t = torch.arange(n, device=DEV).repeat_interleave(dim // 4)
    w = _philox(t, t * 0, torch.arange(dim // 4, device=DEV).repeat(n), t * 0 + 1, seed)
    v = torch.stack([(x >> 8) - (1 << 23) for x in w], 1).double() * 2.0 ** -24 / dim
    return v.view(n, dim)


def _exact_train(case, seed):
    if case["mode"] == "hogwild":
        return None  # the order of the workers' additions is not fixed
    n, dim, K, B, S = (case[k] for k in ("nodes", "dim", "K", "batch", "samples"))
    src, dst, w = _make_graph(case, seed)
    sampler = _Sampler(n, src, dst, w)
    total = 20 * src.numel()
    tables = {}
    for key, t in _train_tables(case, seed, src).items():
        if case["fresh"]:
            f = _fresh_table(n, dim, seed + 1) if key[1] == L.WHICH_U else torch.zeros(n, dim, dtype=torch.float64, device=DEV)
            t = f.float().to(t.dtype)
        tables[key] = t.double()
    for s0 in range(0, S, B * 128):
        t = torch.arange(s0, min(S, s0 + B * 128), device=DEV)
        rec = sampler.records(seed + 7, 0, t, K)
        if case["walk"]:
            rec[:, 0], rec[:, 1] = sampler.walk_pairs(seed + 7, t, case["walk"], case["window"])
        for b0 in range(0, t.numel(), B):
            r = rec[b0:b0 + B]
            eta = LR0 * max(1.0 - (s0 + b0) / total, FLOOR)
            for o in case["orders"]:
                U, C = tables[int(o), L.WHICH_U], tables.get((int(o), L.WHICH_C))
                C = U if C is None else C
                x, c = U[r[:, 0]], C[r[:, 1:]]
                sig = torch.sigmoid(torch.einsum("bd,bkd->bk", x, c))
                g = -eta * case["alpha_neg"] * sig
                g[:, 0] = eta * (1.0 - sig[:, 0])
                dx = torch.einsum("bk,bkd->bd", g, c) - (K + 1) * eta * case["lam"] * x
                dc = g[:, :, None] * x[:, None, :] - eta * case["lam"] * c
                U.index_add_(0, r[:, 0], dx)
                C.index_add_(0, r[:, 1:].reshape(-1), dc.view(-1, dim))
    return [t for _, t in sorted(tables.items())]


def _exact_features(n, dim, src, dst, deg, first, table, known, rows):
    """x of each row: log(1 + degree), then the mean row of its known neighbours, zero padding."""
    P = (dim + 1 + 15) // 16 * 16
    x = torch.zeros(rows.numel(), P, dtype=torch.float64, device=DEV)
    x[:, 0] = torch.log1p(deg[rows])
    lo, cnt = first[rows], first[rows + 1] - first[rows]
    step = 1 << 15
    for i in range(0, rows.numel(), step):
        c = cnt[i:i + step]
        row = torch.repeat_interleave(torch.arange(c.numel(), device=DEV), c)
        arc = torch.arange(row.numel(), device=DEV) - (torch.cumsum(c, 0) - c)[row] + lo[i:i + step][row]
        to = dst[arc]
        ok = known[to]
        row, to = row[ok], to[ok]
        acc = torch.zeros(c.numel(), dim, dtype=torch.float64, device=DEV)
        for k in range(0, row.numel(), 1 << 21):
            acc.index_add_(0, row[k:k + (1 << 21)], table[to[k:k + (1 << 21)]].double())
        num = torch.bincount(row, minlength=c.numel()).clamp(min=1).double()
        x[i:i + step, 1:1 + dim] = acc / num[:, None]
    return x


def _exact_warm(case, seed):
    n, d, H = case["nodes"], case["dim"], case["hidden"]
    src, dst, w, table, known, new, sample = _warm_inputs(case, seed)
    src, dst, new, sample, known = src.long(), dst.long(), new.long(), sample.long(), known.bool()
    first = torch.searchsorted(src, torch.arange(n + 1, device=DEV))
    z = torch.cat([torch.zeros(1, dtype=torch.float64, device=DEV), torch.cumsum(w.double(), 0)])
    deg = z[first[1:]] - z[first[:-1]]
    P = (d + 1 + 15) // 16 * 16
    shapes = ((H, P), (H,), (d, H), (d,))
    flat = torch.arange(sum(math.prod(s) for s in shapes), device=DEV)
    u = ((_words(seed + 9, 7, flat, 1)[0] >> 8) - (1 << 23)).double() * 2.0 ** -23
    p = [t.reshape(s) for t, s in zip(torch.split(u, [math.prod(s) for s in shapes]), shapes)]
    p[0] = p[0] * float(np.float32(1 / math.sqrt(d + 1))) * (torch.arange(P, device=DEV) <= d)
    p[2] = p[2] * float(np.float32(1 / math.sqrt(H)))
    p[1], p[3] = p[1] * 0, p[3] * 0
    p = [t.clone().requires_grad_() for t in p]

    def net(x):
        return torch.nn.functional.gelu(x @ p[0].t() + p[1]) @ p[2].t() + p[3]

    xs = _exact_features(n, d, src, dst, deg, first, table, known, sample)
    ts = table[sample].double()
    m, v, losses = [torch.zeros_like(t) for t in p], [torch.zeros_like(t) for t in p], []
    for s in range(case["steps"]):
        pick = _mulhi(_words(seed + 10, 7, s * case["batch"] + torch.arange(case["batch"], device=DEV), 0), sample.numel())
        loss = torch.nn.functional.mse_loss(net(xs[pick]), ts[pick])
        losses.append(float(loss))
        grads = torch.autograd.grad(loss, p)
        with torch.no_grad():
            for t, g, a, b in zip(p, grads, m, v):
                a.mul_(0.9).add_(g, alpha=0.1)
                b.mul_(0.999).add_(g * g, alpha=0.001)
                t -= 1e-3 * (a / (1 - 0.9 ** (s + 1))) / (torch.sqrt(b / (1 - 0.999 ** (s + 1))) + 1e-8)
    with torch.no_grad():
        y = torch.cat([net(_exact_features(n, d, src, dst, deg, first, table, known, r)) for r in torch.split(new, 1 << 16)])
        return {"losses": losses, "params": torch.cat([t.flatten() for t in p]).cpu().numpy(), "y": y}


def _exact_eval(case, seed):
    n = case["nodes"]
    ksrc, kdst, kw, ps, pd, ns, nd, tables = _eval_inputs(case, seed)
    u, v = torch.cat([ps, ns]).long(), torch.cat([pd, nd]).long()
    scores = []
    for i in range(0, u.numel(), 1 << 20):
        a, b = u[i:i + (1 << 20)], v[i:i + (1 << 20)]
        s, k = 0.0, 0
        for o in (1, 2):
            x, y = tables[o, L.WHICH_U][a].double(), tables[o, L.WHICH_U][b].double()
            t = (x * y).sum(1)
            s = s + (t / (x.norm(dim=1) * y.norm(dim=1)) if case["score"] == "cosine" else t)
            k += 1
        scores.append(s / k if case["score"] == "cosine" else s)
    sampler = _Sampler(n, ksrc, kdst, kw)
    loss = 0.0
    for i in range(0, case["m"], 1 << 17):
        r = sampler.records(seed + 3, 3, torch.arange(i, min(case["m"], i + (1 << 17)), device=DEV), case["K"])
        s = torch.einsum("bd,bkd->bk", tables[2, L.WHICH_U][r[:, 0]].double(), tables[2, L.WHICH_C][r[:, 1:]].double())
        s[:, 1:] *= -1
        loss -= float(torch.nn.functional.logsigmoid(s).sum())
    return {"scores": torch.cat(scores), "auc": None, "counts": None, "loss": loss}


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case["kind"] == "warm":
        return _exact_warm(case, seed)
    if case["kind"] == "eval":
        return _exact_eval(case, seed)
    return None  # alias tables are whole numbers
