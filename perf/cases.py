"""The work that users of this library have it do, as cases to time.

Every case goes through the public entry points of the Python binding (the C
ABI): whole selections on a resident graph, the step-level calls, a batch of
many graphs, a burst of served queries, a first query on a graph that is still
in host memory, the Monte-Carlo spread of a seed set and the estimate + argmax
without allocation.  Graphs are seeded and synthetic (R-MAT 0.57/0.19/0.19,
Erdos-Renyi, Chung-Lu with exponent 2.1), drawn on the GPU, with duplicates and
self-loops removed.
"""
from __future__ import annotations

import ctypes
import math
import random

import numpy as np
import torch

import paper_2410_14047_gb300 as im

DEVICE = "cuda"
M32 = 0xFFFFFFFF
M64 = (1 << 64) - 1

# The schedule the autotuner keeps for a large trivalency graph (edge scans,
# dense walks in vertex order while the frontier is large).
LARGE_SCHEDULE = {"heavy_indeg": 256, "light_batches": 32, "dense_div": 2, "buckets": 0, "pick_tile": 4,
                  "dense_out": 1, "dense_all": 3}


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the smallest plain workload: 10k vertices, 64 simulations, 10 seeds; launches and round trips count
        {"name": "select_er10k", "op": "select", "graph": "er", "n": 10_000, "deg": 10, "model": "uniform",
         "p": 0.01, "J": 64, "K": 10},
        # one graph of the batched workload asked for alone: power law, an odd vertex count
        {"name": "select_chunglu_54k", "op": "select", "graph": "cl", "n": 54_321, "deg": 16, "model": "uniform",
         "p": 0.02, "J": 128, "K": 27},
        # a served query asked for alone, at the widest registers
        {"name": "select_rmat17_j1024", "op": "select", "graph": "rmat", "n": 1 << 17, "deg": 16,
         "model": "uniform", "p": 0.01, "J": 1024, "K": 25},
        # the mid-size plain workload
        {"name": "select_rmat20_wc", "op": "select", "graph": "rmat", "n": 1 << 20, "deg": 16, "model": "wc",
         "p": 0.0, "J": 256, "K": 50},
        # the large plain workload, the benchmark's default, under its schedule
        {"name": "select_rmat24_tri", "op": "select", "graph": "rmat", "n": 1 << 24, "deg": 16,
         "model": "trivalency", "p": 0.0, "J": 512, "K": 50, "schedule": "large"},
        # a caller's own greedy loop over the step-level calls, per-edge weights, a ragged vertex count
        {"name": "steps_explicit_300k", "op": "steps", "graph": "rmat", "n": 300_007, "deg": 16,
         "model": "explicit", "p": 0.0, "J": 256, "K": 3},
        # one sketch and every vertex's estimate sum, no selection (ranking users by influence)
        {"name": "sums_rmat19_tri", "op": "sums", "graph": "rmat", "n": 1 << 19, "deg": 16,
         "model": "trivalency", "p": 0.0, "J": 512, "K": 0},
        # the batched form at an eighth of its graph count: uneven small graphs, J in {64, 128}, K in [5, 50]
        {"name": "batch_64", "op": "batch", "graphs": 64, "n_lo": 1000, "n_hi": 200_000},
        # the served form: a burst of queries of mixed J, K and model on resident graphs of scales 14 to 18
        {"name": "serve_24", "op": "serve", "queries": 24, "scale_lo": 14, "scale_hi": 18, "slots": 8},
        # a first query on a graph that is in host memory: upload, load, selection
        {"name": "cold_rmat21_wc", "op": "cold", "graph": "rmat", "n": 1 << 21, "deg": 16, "model": "wc",
         "p": 0.0, "J": 64, "K": 10},
        # the Monte-Carlo check of a chosen seed set
        {"name": "spread_rmat18_wc", "op": "spread", "graph": "rmat", "n": 1 << 18, "deg": 16, "model": "wc",
         "p": 0.0, "seeds": 50, "R": 1000},
        # estimate + argmax inside a caller's own memory arena, an odd row count
        {"name": "argmax_1m", "op": "argmax", "n": 1_048_573, "J": 256},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_model(rng):
    model = rng.choice(["uniform", "wc", "trivalency", "explicit"])
    return model, (round(rng.uniform(0.005, 0.05), 4) if model == "uniform" else 0.0)


def draw(rng: random.Random):
    op = rng.choice(["select", "select", "select", "select", "steps", "sums", "batch", "serve", "cold", "spread",
                     "argmax"])
    if op == "batch":
        lo = _log_int(rng, 1000, 20_000)
        return {"op": op, "graphs": rng.randint(4, 64), "n_lo": lo, "n_hi": _log_int(rng, 2 * lo, 200_000)}
    if op == "serve":
        lo = rng.randint(14, 16)
        return {"op": op, "queries": rng.randint(2, 24), "scale_lo": lo, "scale_hi": rng.randint(lo, 18),
                "slots": rng.choice([1, 2, 4, 8])}
    if op == "argmax":
        J = rng.choice([16, 64, 128, 256, 512, 1024])
        return {"op": op, "n": _log_int(rng, 1000, (1 << 29) // J), "J": J}
    model, p = _draw_model(rng)
    c = {"op": op, "graph": rng.choice(["rmat", "cl", "er"]), "n": _log_int(rng, 2000, 1 << 20),
         "deg": rng.randint(6, 24), "model": model, "p": p}
    if op == "spread":
        c["n"] = _log_int(rng, 2000, 1 << 18)
        c.update(seeds=rng.randint(1, 50), R=_log_int(rng, 64, 2000))
        return c
    c["J"] = rng.choice([64, 128, 256, 512, 1024])
    while c["n"] * c["J"] > 1 << 28:
        c["J"] //= 2
    c["K"] = {"select": rng.randint(5, 50), "cold": rng.randint(5, 50), "steps": rng.randint(1, 4), "sums": 0}[op]
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(int(seed) & ((1 << 63) - 1))
    return g


def _csr(u, v, n):
    """Host CSR (int32) of the distinct edges u -> v without self-loops."""
    keep = u != v
    key = torch.unique(u[keep] * n + v[keep])
    u = torch.div(key, n, rounding_mode="floor")
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=key.device)
    rowptr[1:] = torch.cumsum(torch.bincount(u, minlength=n), 0)
    col = (key - u * n).to(torch.int32)
    return rowptr.to(torch.int32).cpu().numpy(), col.cpu().numpy()


def _graph(kind, n, deg, seed):
    gen = _gen(seed)
    draws = n * deg
    if kind == "er":
        u = torch.randint(0, n, (draws,), generator=gen, device=DEVICE)
        v = torch.randint(0, n, (draws,), generator=gen, device=DEVICE)
        return _csr(u, v, n)
    if kind == "cl":
        # weights (i + i0)^(-1/1.1), i0 such that the largest expected degree is about sqrt(edges)
        i = torch.arange(n, dtype=torch.float64, device=DEVICE)
        lo, hi = 1.0, float(n)
        for _ in range(30):
            i0 = math.sqrt(lo * hi)
            w = (i + i0) ** (-1.0 / 1.1)
            if float(w[0] / w.sum()) > 1.0 / math.sqrt(draws):
                lo = i0
            else:
                hi = i0
        cum = torch.cumsum(w, 0)
        cum /= cum[-1].clone()
        u = torch.searchsorted(cum, torch.rand(draws, generator=gen, device=DEVICE, dtype=torch.float64))
        v = torch.searchsorted(cum, torch.rand(draws, generator=gen, device=DEVICE, dtype=torch.float64))
        return _csr(u.clamp_(max=n - 1), v.clamp_(max=n - 1), n)
    scale = max(1, (n - 1).bit_length())
    u = torch.zeros(draws, dtype=torch.int64, device=DEVICE)
    v = torch.zeros(draws, dtype=torch.int64, device=DEVICE)
    for _ in range(scale):
        r = torch.rand(draws, generator=gen, device=DEVICE)
        u = (u << 1) | (r >= 0.76)
        v = (v << 1) | (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    if n < 1 << scale:  # ids past an odd vertex count are dropped
        keep = (u < n) & (v < n)
        u, v = u[keep], v[keep]
    return _csr(u, v, n)


def _model(case, m, seed):
    kind = case["model"]
    if kind == "uniform":
        return {"kind": "uniform", "p": case["p"]}
    if kind == "trivalency":
        return {"kind": "trivalency", "seed": int(seed)}
    if kind == "explicit":
        w = torch.randn(m, generator=_gen(seed + 1), device=DEVICE).mul_(0.025).add_(0.05).clamp_(0.0, 1.0)
        return {"kind": "explicit", "w": w.cpu().numpy()}
    return {"kind": "wc"}


def _batch_inputs(case, seed):
    rng = random.Random(seed)
    graphs, p, J, K = [], [], [], []
    for g in range(case["graphs"]):
        rp, col = _graph("cl", rng.randint(case["n_lo"], case["n_hi"]), rng.randint(8, 32), seed * 1000 + g)
        graphs.append(_HostGraph(rp, col))
        p.append(rng.uniform(0.005, 0.05))
        J.append(rng.choice([64, 128]))
        K.append(5 + (17 * g) % 46)  # 5 to 50, the same for every seed: so many seeds come back
    return graphs, np.array(p, np.float32), np.array(J, np.int32), np.array(K, np.int32)


def _ranks(case, seed):
    """Registers as a sketch holds them: geometric ranks, a few visited marks."""
    gen, n, J = _gen(seed), case["n"], case["J"]
    M = torch.empty(n * J, dtype=torch.uint8, device=DEVICE)
    step = 1 << 26
    for a in range(0, n * J, step):
        b = min(n * J, a + step)
        r = torch.rand(b - a, generator=gen, device=DEVICE)
        rank = torch.floor(-torch.log2(r.clamp_(min=2.0 ** -31))).to(torch.uint8)
        M[a:b] = torch.where(r > 0.999, torch.full_like(rank, 0xFF), rank)
    return M


class _HostGraph:
    def __init__(self, rowptr, col):
        self.rowptr, self.col = rowptr, col


def prepare(case, seed):
    op = case["op"]
    st = {"op": op, "case": case, "seed": int(seed)}
    if op == "argmax":
        n = case["n"]
        st["M"] = _ranks(case, seed)
        st["picked"] = torch.zeros((n + 31) // 32, dtype=torch.int32, device=DEVICE)
        st["s"] = torch.zeros(1, dtype=torch.int32, device=DEVICE)
        st["S"] = torch.zeros(1, dtype=torch.int64, device=DEVICE)
        st["est"] = torch.zeros(1, dtype=torch.float64, device=DEVICE)
        st["stream"] = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream or None)
        st["lib"] = im.load_library()
        return st
    ctx = im.im_ctx_create(0)
    st["ctx"] = ctx
    if op == "batch":
        graphs, p, J, K = _batch_inputs(case, seed)
        st.update(batch=im.im_batch_load(ctx, graphs, p), J=J, K=K)
        return st
    if op == "serve":
        rng = random.Random(seed)
        srv = im.Server(0, slots=case["slots"])
        scales = list(range(case["scale_lo"], case["scale_hi"] + 1))
        for i, s in enumerate(scales):
            rp, col = _graph("rmat", 1 << s, 16, seed * 100 + i)
            srv.add_graph(im.im_graph_load(ctx, rp, col, {"kind": "wc"}))
        # every graph, K, J and kind of model comes up in turn, the simulation seeds are drawn
        st["queries"] = [{"graph": i % len(scales), "K": (10, 25, 50)[i // 3 % 3], "J": (64, 256, 1024)[i % 3],
                          "model": {"kind": "wc"} if i % 2 else {"kind": "uniform", "p": 0.01},
                          "seed": rng.getrandbits(40), "rebuild_eps": 0.01} for i in range(case["queries"])]
        st["server"] = srv
        return st
    rp, col = _graph(case["graph"], case["n"], case["deg"], seed)
    model = _model(case, col.shape[0], seed)
    if case.get("schedule") == "large":
        im.im_ctx_set_tuning(ctx, LARGE_SCHEDULE)
    if op == "cold":
        st.update(rowptr=rp, col=col, model=model)
        return st
    st["graph"] = im.im_graph_load(ctx, rp, col, model)
    if op == "spread":
        # the seeds of an influence maximization are high-degree vertices: the k of largest out-degree
        st["seeds"] = np.argsort(-np.diff(rp), kind="stable")[: case["seeds"]].astype(np.int32)
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _joined(results):
    return {k: np.concatenate([r[k] for r in results]) for k in ("seeds", "score", "est")}


def run(st):
    op, case, seed = st["op"], st["case"], st["seed"]
    if op == "select":
        return im.im_select_seeds(st["graph"], case["K"], case["J"], seed=seed)
    if op == "cold":
        g = im.im_graph_load(st["ctx"], st["rowptr"], st["col"], st["model"])
        r = im.im_select_seeds(g, case["K"], case["J"], seed=seed)
        g.free()
        return r
    if op == "sums":
        sk = im.im_sketch_build(st["graph"], case["J"], seed)
        S = sk.sums()
        sk.free()
        return S.view(np.int64)
    if op == "steps":
        sk = im.im_sketch_build(st["graph"], case["J"], seed)
        picks, counts = [], []
        for _ in range(case["K"]):
            picks.append(sk.pick())
            counts.append(sk.cover(picks[-1][0]))
            sk.rebuild()
        S = sk.sums()
        sk.free()
        return {"seeds": np.array([p[0] for p in picks], np.int32), "S": np.array([p[1] for p in picks], np.int64),
                "est": np.array([p[2] for p in picks]), "counts": np.array(counts, np.int64),
                "sums": S.view(np.int64)}
    if op == "batch":
        return _joined(im.im_batch_select_seeds(st["batch"], st["J"], st["K"], seed=seed))
    if op == "serve":
        tickets = [st["server"].submit(**q) for q in st["queries"]]
        results = [st["server"].wait(t) for t in tickets]
        if any(r["status"] for r in results):
            raise RuntimeError(next(r["error"] for r in results if r["status"]))
        return _joined(results)
    if op == "spread":
        return im.im_spread_mc(st["graph"], st["seeds"], case["R"], seed=seed)
    rc = st["lib"].im_argmax_noalloc(st["M"].data_ptr(), case["n"], case["J"], st["picked"].data_ptr(),
                                     st["stream"], st["s"].data_ptr(), st["S"].data_ptr(), st["est"].data_ptr())
    if rc:
        raise RuntimeError(im.STATUS.get(rc, rc))
    return [st["s"], st["S"], st["est"], st["picked"]]


def work(case):
    """Bytes one pass cannot do without: the CSR read once, every register
    written once and read once by an estimate, the results written; flops: one
    rank a register (spread: one reached mark a vertex and simulation)."""
    op = case["op"]
    if op == "argmax":
        return {"bytes": case["n"] * case["J"] + case["n"] / 8, "flops": case["n"] * case["J"]}
    if op == "batch":
        n = case["graphs"] * (case["n_lo"] + case["n_hi"]) / 2
        return {"bytes": n * (4 + 4 * 20) + 2 * n * 96, "flops": n * 96}
    if op == "serve":
        scales = range(case["scale_lo"], case["scale_hi"] + 1)
        n = case["queries"] * sum(1 << s for s in scales) / len(scales)
        return {"bytes": n * (4 + 4 * 16) + 2 * n * 448, "flops": n * 448}
    n, m = case["n"], case["n"] * case["deg"]
    csr = 4 * (n + m) + (4 * m if case["model"] == "explicit" else 0)
    if op == "spread":
        return {"bytes": csr + n * case["R"] / 8, "flops": n * case["R"]}
    return {"bytes": csr + 2 * n * case["J"], "flops": n * case["J"]}


# ---------------------------------------------------------------------------
# the same results in plain 64-bit arithmetic
# ---------------------------------------------------------------------------

def _splitmix(seed, k):
    z = (seed + (k + 1) * 0x9E3779B97F4A7C15) & M64
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & M64
    return z ^ (z >> 31)


def _mul(x, c):
    return (x * c) & M32


def _rotl(x, r):
    return ((x << r) | (x >> (32 - r))) & M32


def _mm3(words, seed, length):
    """MurmurHash3_x86_32 of whole 4-byte words held in int64 tensors."""
    h = seed
    for k in words:
        h = h ^ _mul(_rotl(_mul(k, 0xCC9E2D51), 15), 0x1B873593)
        h = (_mul(_rotl(h, 13), 5) + 0xE6546B64) & M32
    h = h ^ length
    h = _mul(h ^ (h >> 16), 0x85EBCA6B)
    h = _mul(h ^ (h >> 13), 0xC2B2AE35)
    return h ^ (h >> 16)


def _threshold(w):
    return torch.floor(w.double() * 2147483648.0).to(torch.int64)


def _edges(rp, col):
    n = rp.shape[0] - 1
    deg = torch.from_numpy(np.diff(rp)).to(DEVICE, torch.int64)
    u = torch.repeat_interleave(torch.arange(n, device=DEVICE), deg)
    return u, torch.from_numpy(col).to(DEVICE, torch.int64)


def _thresholds(u, v, n, model):
    kind = model["kind"]
    if kind == "uniform":
        return _threshold(torch.tensor(model["p"], dtype=torch.float32)).to(DEVICE).expand(u.shape)
    if kind == "wc":
        indeg = torch.bincount(v, minlength=n).to(torch.float32)
        return _threshold(torch.ones_like(indeg) / indeg.clamp(min=1))[v]
    if kind == "explicit":
        return _threshold(torch.from_numpy(model["w"]).to(DEVICE))
    s = model["seed"]
    cls = _mm3([u, v], (s ^ (s >> 32)) & M32, 8) % 3
    return _threshold(torch.tensor([0.1, 0.01, 0.001], dtype=torch.float32)).to(DEVICE)[cls]


def _sims(J, seed):
    z = [_splitmix(seed, j) for j in range(J)]
    order = sorted(range(J), key=lambda j: z[j] & 0x7FFFFFFF)
    X = torch.tensor([z[j] & 0x7FFFFFFF for j in order], device=DEVICE)
    return X, torch.tensor([z[j] >> 32 for j in order], device=DEVICE)


def _greedy(rp, col, model, K, J, seed, eps=0.01):
    """The selection by its definition: ranks, fixpoint, estimate, cover, rebuild rule."""
    n = rp.shape[0] - 1
    u, v = _edges(rp, col)
    X, salt = _sims(J, seed)
    thr = _thresholds(u, v, n, model)
    live = (X[None, :] ^ (_mm3([u, v], 0, 8) & 0x7FFFFFFF)[:, None]) < thr[:, None]
    h = _mm3([torch.arange(n, device=DEVICE)[:, None]], salt[None, :], 4)
    rank = (32 - torch.frexp(h.double())[1]).to(torch.int32)
    ui, vi = u[:, None].expand(-1, J), v[:, None].expand(-1, J)
    vis = torch.zeros(n, J, dtype=torch.bool, device=DEVICE)

    def fixpoint():
        M = rank.clone()
        while True:
            from_v = torch.where(live & ~vis[v], M[v], torch.zeros((), dtype=M.dtype, device=DEVICE))
            new = M.scatter_reduce(0, ui, from_v, "amax") if u.numel() else M
            new = torch.where(vis, rank, new)
            if torch.equal(new, M):
                return M
            M = new

    M, picked = fixpoint(), torch.zeros(n, dtype=torch.bool, device=DEVICE)
    seeds, score, est, old = [], [], [], 0
    for k in range(K):
        S = torch.where(vis, 1 << 32, torch.ones_like(M, dtype=torch.int64) << (32 - M.long())).sum(1)
        least = S[~picked].min()
        s = int(torch.nonzero((S == least) & ~picked)[0])
        picked[s] = True
        front = torch.zeros_like(vis)
        front[s] = ~vis[s]
        vis = vis | front
        while u.numel() and bool(front.any()):
            hit = torch.zeros(n, J, dtype=torch.int32, device=DEVICE)
            hit.scatter_reduce_(0, vi, (live & front[u]).to(torch.int32), "amax")
            front = (hit > 0) & ~vis
            vis = vis | front
        count = int(vis.sum())
        seeds.append(s)
        score.append(count / J)
        est.append(J * 4294967296.0 / (0.77351 * int(least)))
        if k + 1 < K and (count / J - old / J) / (count / J) > eps:
            M, old = fixpoint(), count
    return {"seeds": np.array(seeds, np.int32), "score": np.array(score), "est": np.array(est)}


def _spread(rp, col, model, seeds, R, seed):
    """Independent-cascade spread with one coin a simulation and edge: (seed stream output r m + e) >> 33 < thr[e]."""
    n, m = rp.shape[0] - 1, col.shape[0]
    u, v = _edges(rp, col)
    thr = _thresholds(u, v, n, model)
    s64 = lambda x: x - (1 << 64) if x >> 63 else x  # noqa: E731
    shr = lambda z, k: (z >> k) & ((1 << (64 - k)) - 1)  # noqa: E731
    e = torch.arange(m, device=DEVICE)
    reach = []
    step = max(1, (1 << 26) // max(m, 1))
    for r0 in range(0, R, step):
        r = torch.arange(r0, min(R, r0 + step), device=DEVICE)
        z = s64(seed & M64) + (r[None, :] * m + e[:, None] + 1) * s64(0x9E3779B97F4A7C15)
        z = (z ^ shr(z, 30)) * s64(0xBF58476D1CE4E5B9)
        z = (z ^ shr(z, 27)) * s64(0x94D049BB133111EB)
        live = shr(z ^ shr(z, 31), 33) < thr[:, None]
        vis = torch.zeros(n, r.numel(), dtype=torch.bool, device=DEVICE)
        vis[torch.from_numpy(np.asarray(seeds)).to(DEVICE, torch.int64)] = True
        front, vi = vis, v[:, None].expand(-1, r.numel())
        while m and bool(front.any()):
            hit = torch.zeros(n, r.numel(), dtype=torch.int32, device=DEVICE)
            hit.scatter_reduce_(0, vi, (live & front[u]).to(torch.int32), "amax")
            front = (hit > 0) & ~vis
            vis = vis | front
        reach += vis.sum(0).tolist()
    total, sq = sum(reach), sum(x * x for x in reach)
    var = (sq - total * total / R) / (R - 1)
    return {"mean": total / R, "stderr": math.sqrt(max(var, 0.0) / R), "sum": total, "sumsq": sq}


def exact(case, seed):
    op = case["op"]
    if op == "argmax":
        M = _ranks(case, seed).view(case["n"], case["J"])
        S = torch.empty(case["n"], dtype=torch.int64, device=DEVICE)
        for a in range(0, case["n"], 1 << 16):
            r = M[a:a + (1 << 16)].long()
            S[a:a + (1 << 16)] = torch.where(r == 0xFF, 1 << 32, 1 << (32 - r.clamp(max=32))).sum(1)
        least = S.min()
        s = torch.nonzero(S == least)[:1, 0]
        return [s.to(torch.int32), least[None], case["J"] * 4294967296.0 / (0.77351 * least[None].double()), None]
    if op in ("select", "cold", "spread"):
        if case["n"] * case["deg"] * case.get("J", case.get("R", 0)) > (6 << 30 if op == "spread" else 1 << 27):
            return None
        rp, col = _graph(case["graph"], case["n"], case["deg"], seed)
        model = _model(case, col.shape[0], seed)
        if op == "spread":
            k = np.argsort(-np.diff(rp), kind="stable")[: case["seeds"]]
            return _spread(rp, col, model, k, case["R"], int(seed))
        return _greedy(rp, col, model, case["K"], case["J"], int(seed))
    return None  # whole numbers (sums), or selections too large for the plain form
