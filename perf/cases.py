"""The work users have this library do, as timed cases over the public API.

A case is one call (or one short sequence of calls) a program makes: loading
a graph and building its tables, estimating from a resident graph, counting a
shard of a sample range, turning summed counts into estimates, running a batch
of requests over many graphs, serving a burst of requests.  The graphs are
the kinds the repository's workloads name: Chung-Lu graphs with power-law
expected degrees and 2-D random geometric graphs on the unit torus, generated
here on the GPU from the seed alone.

`prepare` makes what a program holds before the call (the CSR on the device,
or the loaded graph, batch or server); `run` is the call; `work` the bytes
and operations it cannot do without; `exact` the outputs in plain 64-bit
numpy where they are functions of the inputs alone.  Sampled counts have no
such value: they depend on the random words.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1509_08089_gb300 as moss

DEVICE = "cuda"
K4, K5, MIN = 1 << 4, 1 << 5, moss.TABLES_4MIN


# ------------------------------------------------------------------ graphs --
def _csr(a: torch.Tensor, b: torch.Tensor, n: int):
    """(row_ptr int64[n+1], col int32[nnz]) of the simple undirected graph
    with edges {a_i, b_i}: loops and repeated edges dropped, lists sorted."""
    keep = a != b
    a, b = a[keep], b[keep]
    key = torch.unique(torch.minimum(a, b) * n + torch.maximum(a, b))
    lo, hi = torch.div(key, n, rounding_mode="floor"), key % n
    both = torch.sort(torch.cat([key, hi * n + lo])).values
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=both.device)
    deg = torch.bincount(torch.div(both, n, rounding_mode="floor"), minlength=n)
    torch.cumsum(deg, 0, out=row_ptr[1:])
    return row_ptr, (both % n).to(torch.int32)


def chung_lu(n: int, gamma: float, dbar: float, dmax: float, seed: int):
    """Expected degrees w_i = c (i + i0)^-a, a = 1 / (gamma - 1), i0 such that
    the largest is about dmax at mean dbar: n dbar / 2 edges with both ends
    drawn in proportion to w, the vertices in random order."""
    a = 1.0 / (gamma - 1.0)

    def top(i0):   # w_0 for this shift
        if abs(a - 1.0) < 1e-9:
            mass = math.log((n + i0) / i0)
        else:
            mass = ((n + i0) ** (1.0 - a) - i0 ** (1.0 - a)) / (1.0 - a)
        return dbar * n * i0 ** -a / mass

    lo, hi = 1e-6, float(n)
    for _ in range(80):
        mid = math.sqrt(lo * hi)
        lo, hi = (mid, hi) if top(mid) > dmax else (lo, mid)
    i0 = hi
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    m = int(n * dbar / 2)

    def ends():
        u = torch.rand(m, generator=gen, device=DEVICE, dtype=torch.float64)
        if abs(a - 1.0) < 1e-9:
            x = i0 * torch.exp(u * math.log((n + i0) / i0))
        else:
            e0, e1 = i0 ** (1.0 - a), (n + i0) ** (1.0 - a)
            x = (e0 + u * (e1 - e0)) ** (1.0 / (1.0 - a))
        return (x - i0).to(torch.int64).clamp_(0, n - 1)

    perm = torch.randperm(n, generator=gen, device=DEVICE)
    return _csr(perm[ends()], perm[ends()], n)


def geometric(n: int, dbar: float, seed: int):
    """Points of the unit torus joined within r = sqrt(dbar / (pi n)), in
    random order: nearly equal degrees, many triangles."""
    r = math.sqrt(dbar / (math.pi * n))
    g = max(3, int(1.0 / r))   # cells of side >= r
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    x, y = torch.rand(2, n, generator=gen, device=DEVICE, dtype=torch.float64)
    cx, cy = (x * g).to(torch.int64).clamp_(0, g - 1), (y * g).to(torch.int64).clamp_(0, g - 1)
    cell, order = torch.sort(cx * g + cy)
    start = torch.zeros(g * g + 1, dtype=torch.int64, device=DEVICE)
    torch.cumsum(torch.bincount(cell, minlength=g * g), 0, out=start[1:])
    most = int((start[1:] - start[:-1]).max())
    xs, ys, cx, cy = x[order], y[order], cx[order], cy[order]
    i = torch.arange(n, device=DEVICE)
    src, dst = [], []
    for dx, dy in ((0, 0), (0, 1), (1, -1), (1, 0), (1, 1)):   # each pair of cells once
        other = (cx + dx) % g * g + (cy + dy) % g
        for k in range(most):
            j = start[other] + k
            ok = j < start[other + 1]
            if (dx, dy) == (0, 0):
                ok &= j > i
            a, b = i[ok], j[ok]
            ex, ey = (xs[a] - xs[b]).abs(), (ys[a] - ys[b]).abs()
            ex, ey = torch.minimum(ex, 1.0 - ex), torch.minimum(ey, 1.0 - ey)
            near = ex * ex + ey * ey <= r * r
            src.append(a[near])
            dst.append(b[near])
    return _csr(order[torch.cat(src)], order[torch.cat(dst)], n)


def _graph(case: dict, seed: int):
    if case["graph"] == "geometric":
        return geometric(case["n"], case["dbar"], seed)
    return chung_lu(case["n"], case["gamma"], case["dbar"], case["dmax"], seed)


def _specs(case: dict, seed: int):
    """Graphs and requests of a batch: n log-uniform in [500, n], every other
    one geometric, k 4 or 5 and a budget log-uniform in [1e4, budget]."""
    rng = np.random.default_rng(seed)
    out = []
    for i in range(case["graphs"]):
        n = int(math.exp(rng.uniform(math.log(500), math.log(case["n"]))))
        if i % 2 == 0:
            dbar = float(rng.uniform(4.0, 12.0))
            g = {"graph": "chung_lu", "n": n, "gamma": float(rng.uniform(2.0, 3.0)), "dbar": dbar,
                 "dmax": min(0.2 * n, 50 * dbar)}
        else:
            g = {"graph": "geometric", "n": n, "dbar": float(rng.uniform(6.0, 30.0))}
        k = int(rng.choice([4, 5]))
        budget = int(math.exp(rng.uniform(math.log(1e4), math.log(case["budget"]))))
        out.append((g, k, budget, int(rng.integers(1, 2**62)), seed * 1000 + i))
    return out


# ------------------------------------------------------------------- cases --
def listed() -> list[dict]:
    big = {"graph": "chung_lu", "n": 4_000_000, "gamma": 2.1, "dbar": 17.0, "dmax": 20_000.0}
    mid = {"graph": "chung_lu", "n": 100_000, "gamma": 2.2, "dbar": 20.0, "dmax": 5_000.0}
    small = {"graph": "chung_lu", "n": 2_000, "gamma": 2.5, "dbar": 8.0, "dmax": 200.0}
    return [
        # counts summed over the shards of a split run, made into estimates and their covariances
        {"name": "finalize_shards", "do": "finalize", **mid, "budget": 10**9},
        # an interactive question about a small resident graph: all latency
        {"name": "estimate_small", "do": "estimate", **small, "k": 4, "budget": 100_000, "order": "input",
         "rng": "splitmix"},
        # a small graph arrives, one answer is wanted, the graph goes
        {"name": "oneshot_small", "do": "step", **small, "n": 5_003, "tables": "5", "budget": 100_001,
         "order": "input"},
        # a mesh-like resident graph: equal degrees, many triangles, an odd budget
        {"name": "estimate_mesh", "do": "estimate", "graph": "geometric", "n": 300_007, "dbar": 13.0, "k": 5,
         "budget": 5_000_011, "order": "input", "rng": "splitmix"},
        # one rank's share of a split Path-5 run on a graph of several million edges: an odd range of ids
        {"name": "shard_counts", "do": "counts", "graph": "chung_lu", "n": 1_000_003, "gamma": 2.3, "dbar": 14.0,
         "dmax": 8_000.0, "method": 2, "first": 123_457, "budget": 25_000_001, "order": "degree"},
        # the five-node step at one million edges: load, tables, 1e8 samples, estimates
        {"name": "step_1m", "do": "step", **mid, "tables": "5", "budget": 10**8, "order": "input"},
        # the four-node mix (MOSS-4 and MOSS-4Min) at one million edges, tables included
        {"name": "mix_1m", "do": "step", **mid, "tables": "4min", "budget": 4 * 10**7, "order": "input"},
        # every table of a graph of several million edges, with a pilot's worth of samples
        {"name": "onboard_large", "do": "step", "graph": "chung_lu", "n": 1_000_000, "gamma": 2.2, "dbar": 16.0,
         "dmax": 15_000.0, "tables": "all", "budget": 40_000, "order": "degree"},
        # four-node estimate of the resident 34M-edge graph in its own ids, Philox words
        {"name": "estimate_34m_k4", "do": "estimate", **big, "k": 4, "budget": 3 * 10**8, "order": "input",
         "rng": "philox"},
        # the five-node step at 34 million edges: the largest
        {"name": "step_34m", "do": "step", **big, "tables": "5", "budget": 10**9, "order": "degree"},
        # requests of uneven size over many resident graphs in one launch
        {"name": "batch_many", "do": "batch", "graphs": 256, "n": 50_000, "budget": 10**7},
        # a burst of requests with target errors at a server holding 12 graphs
        {"name": "serve_burst", "do": "serve", "graphs": 12, "edges": 1_000_000, "requests": 64},
    ]


def draw(rng) -> dict:
    """One more case of the same kinds and ranges."""
    def log(lo, hi):
        return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))

    def power(n):
        dbar = rng.uniform(6.0, 20.0)
        return {"graph": "chung_lu", "n": n, "gamma": rng.uniform(2.1, 2.8), "dbar": dbar,
                "dmax": float(min(0.1 * n, rng.uniform(100.0, 20_000.0)))}

    do = rng.choice(["finalize", "estimate", "estimate", "counts", "step", "step", "batch", "serve"])
    if do == "finalize":
        return {"do": do, **power(log(2_000, 200_000)), "budget": log(10**5, 10**10)}
    if do == "batch":
        return {"do": do, "graphs": log(4, 256), "n": log(2_000, 50_000), "budget": log(10**5, 10**7)}
    if do == "serve":
        return {"do": do, "graphs": log(2, 12), "edges": log(50_000, 1_000_000), "requests": log(4, 64)}
    n = log(2_000, 3_500_000)
    graph = power(n)
    if n <= 400_000 and rng.random() < 0.3:
        graph = {"graph": "geometric", "n": n, "dbar": rng.uniform(6.0, 20.0)}
    most = 3 * 10**8
    order = rng.choice(["input", "degree"])
    if do == "counts":
        return {"do": do, **graph, "method": rng.choice([0, 1, 2, 3]), "first": log(1, 10**9),
                "budget": log(10**4, most), "order": order}
    if do == "estimate":
        return {"do": do, **graph, "k": rng.choice([4, 5]), "budget": log(10**4, most), "order": order,
                "rng": rng.choice(["splitmix", "splitmix", "philox"])}
    return {"do": do, **graph, "tables": rng.choice(["4", "5", "4min", "all"]), "budget": log(10**4, most),
            "order": order}


# ----------------------------------------------------------------- prepare --
_ORDERS = {"input": moss.ORDER_INPUT, "degree": moss.ORDER_DEGREE}
_RNGS = {"splitmix": moss.RNG_SPLITMIX64, "philox": moss.RNG_PHILOX4X32}
_MASKS = {"4": K4, "5": K5, "4min": K4 | MIN, "all": K4 | K5 | MIN}


def _shard_counts(case: dict, seed: int):
    """K and hits of a split five-node run: every sample in one class that its
    sub-method can see, most in the sparse ones."""
    rng = np.random.default_rng(seed)
    K = (case["budget"] // 2, case["budget"] - case["budget"] // 2)
    hits = np.zeros((2, 22), dtype=np.uint64)
    for l in range(2):
        share = 4.0 ** -np.sqrt(np.arange(22.0)) * rng.uniform(0.5, 1.5, 22)
        share[1:] *= _PHI5[:, l] > 0
        hits[l] = rng.multinomial(K[l], share / share.sum())
    return np.array(K, dtype=np.uint64), hits


def prepare(case: dict, seed: int) -> dict:
    do = case["do"]
    if do == "batch":
        batch, graphs = moss.Batch(), []
        for g, k, budget, sample_seed, graph_seed in _specs(case, seed):
            graphs.append(moss.Graph(*_graph(g, graph_seed)))
            batch.add(graphs[-1], k, budget, sample_seed)
        return {"case": case, "batch": batch, "graphs": graphs}
    if do == "serve":
        rng = np.random.default_rng(seed)
        server, graphs = moss.Server(), []
        for i in range(case["graphs"]):
            edges = math.exp(rng.uniform(math.log(1e4), math.log(case["edges"])))
            dbar = float(rng.uniform(8.0, 20.0))
            n = max(200, int(2 * edges / dbar))
            graphs.append(moss.Graph(*chung_lu(n, float(rng.uniform(2.1, 2.8)), dbar, min(0.2 * n, 50 * dbar),
                                               seed * 1000 + i)))
            server.add_graph(graphs[-1])
        requests = [(int(rng.integers(0, case["graphs"])), int(rng.choice([4, 5])), float(rng.uniform(0.01, 0.05)),
                     int(rng.integers(1, 2**62))) for _ in range(case["requests"])]
        return {"case": case, "server": server, "graphs": graphs, "requests": requests}
    row_ptr, col = _graph(case, seed)
    if do == "step":
        return {"case": case, "row_ptr": row_ptr, "col": col, "seed": seed}
    order = _ORDERS[case.get("order", "input")]
    if do == "finalize":
        K, hits = _shard_counts(case, seed)
        return {"case": case, "graph": moss.Graph(row_ptr, col, k_mask=K5), "K": K, "hits": hits}
    if do == "counts":
        mask = MIN if case["method"] == 3 else K4 if case["method"] == 0 else K5
        return {"case": case, "graph": moss.Graph(row_ptr, col, k_mask=mask, order=order), "seed": seed,
                "counts": torch.zeros(22, dtype=torch.int64, device=DEVICE)}
    return {"case": case, "graph": moss.Graph(row_ptr, col, k_mask=1 << case["k"], order=order,
                                              rng=_RNGS[case["rng"]]), "seed": seed}


# --------------------------------------------------------------------- run --
def _stack(results: list[dict]) -> dict:
    """Many results with one array per field."""
    return {f: np.stack([np.asarray(r[f]) for r in results]) for f in results[0]}


def run(state: dict):
    case = state["case"]
    do = case["do"]
    if do == "estimate":
        return state["graph"].estimate(case["k"], case["budget"], state["seed"])
    if do == "counts":
        moss.moss_sample_counts(state["graph"].handle, case["method"], case["first"], case["budget"], state["seed"],
                                state["counts"])
        return state["counts"]
    if do == "finalize":
        cov, result = moss.moss_covariance(state["graph"].handle, 5, state["K"], state["hits"])
        return {"cov": cov, **result}
    if do == "batch":
        return _stack(state["batch"].run())
    if do == "serve":
        server = state["server"]
        ids = [server.submit(g, k, target_rse=eps, seed=s) for g, k, eps, s in state["requests"]]
        return _stack([server.wait(i)[0] for i in ids])
    # do == "step": from the CSR to the estimates and the graph's exact totals
    with moss.Graph(state["row_ptr"], state["col"], k_mask=_MASKS[case["tables"]],
                    order=_ORDERS[case["order"]]) as g:
        B, out = case["budget"], {}
        if case["tables"] in ("4min", "all"):
            out["mix"] = g.estimate_min(B // 2, B - B // 2, state["seed"])
        if case["tables"] in ("4", "5"):
            out["estimate"] = g.estimate(int(case["tables"]), B, state["seed"])
        elif case["tables"] == "all":
            out["estimate"] = g.estimate(5, B, state["seed"])
        s = g.stats()
        out["totals"] = {"gamma": np.array(list(s.gamma_d)[:3]), "lambda3": s.lambda3_d, "lambda4": s.lambda4_d,
                         "d_max": int(s.d_max)}
        return out


# -------------------------------------------------------------------- work --
def _edges(case: dict) -> float:
    return case["n"] * case["dbar"] / 2


def _csr_bytes(case: dict) -> float:
    return 8.0 * (case["n"] + 1) + 8.0 * _edges(case)


#: random words a sample reads, and pairs it has to test for an edge
_WORDS = {0: 6, 1: 7, 2: 8, 3: 6}
_PAIRS = {0: 3, 1: 6, 2: 6, 3: 3}
_OPS_WORD, _OPS_PAIR = 11, 8   # the operations of one word and its index product; of one key and its comparison
_RESULT = 8.0 * 270


def _sampling(method: int, count: float, table_bytes: float):
    """A sample's ids (4 bytes each) come from the resident graph, which need
    not be read more than once."""
    ids = {0: 4, 1: 5, 2: 5, 3: 4}[method]
    return (min(4.0 * ids * count, table_bytes), count * (_WORDS[method] * _OPS_WORD + _PAIRS[method] * _OPS_PAIR))


def work(case: dict) -> dict:
    do = case["do"]
    if do == "finalize":
        return {"bytes": 8.0 * (2 + 44 + 22 * 22) + _RESULT, "flops": 2.0 * 22 * 22 * 5}
    if do in ("batch", "serve"):
        # means of the distributions that the requests are drawn from
        if do == "batch":
            n = (case["n"] - 500) / math.log(case["n"] / 500) if case["n"] > 500 else 500.0
            per = (case["budget"] - 1e4) / math.log(case["budget"] / 1e4)
            count, table = case["graphs"], case["graphs"] * n * 13.0 * 4
        else:
            e = (case["edges"] - 1e4) / math.log(case["edges"] / 1e4)
            count, table, per = case["requests"], case["graphs"] * e * 8.0, 2e5
        b, f = _sampling(1, count * per, table)
        return {"bytes": b + count * _RESULT, "flops": f}
    table = _csr_bytes(case)
    if do == "counts":
        b, f = _sampling(case["method"], case["budget"], table)
        return {"bytes": b + 8.0 * 22, "flops": f}
    if do == "estimate":
        parts = [(0, case["budget"])] if case["k"] == 4 else [(1, case["budget"] / 2), (2, case["budget"] / 2)]
        f = sum(_sampling(m, c, table)[1] for m, c in parts)
        return {"bytes": min(sum(_sampling(m, c, table)[0] for m, c in parts), table) + _RESULT, "flops": f}
    half = case["budget"] / 2
    parts = {"4": [(0, 2 * half)], "5": [(1, half), (2, half)], "4min": [(0, half), (3, half)],
             "all": [(0, half), (3, half), (1, half), (2, half)]}[case["tables"]]
    f = sum(_sampling(m, c, table)[1] for m, c in parts)
    # the exact vertex weights: a product and a sum or two for each slot and vertex
    return {"bytes": table + _RESULT, "flops": f + 4.0 * 2 * _edges(case) + 20.0 * case["n"]}


# ------------------------------------------------------------------- exact --
#: Table 2 of arXiv 1509.08089: forks, 5-paths and 4-stars in each five-node class
_PHI5 = np.array([
    [0, 1, 0], [0, 0, 1], [1, 0, 0], [1, 2, 0], [2, 2, 0], [0, 5, 0], [2, 1, 0], [2, 0, 1], [4, 4, 0], [4, 7, 0],
    [5, 2, 1], [4, 4, 1], [6, 6, 0], [10, 10, 1], [9, 6, 1], [12, 6, 2], [10, 14, 0], [20, 24, 1], [20, 18, 2],
    [36, 36, 3], [60, 60, 5]], dtype=np.float64)


def _totals(row_ptr: torch.Tensor, col: torch.Tensor):
    """(Gamma, Gamma1, Gamma2), Lambda3, Lambda4, d_max as exact integers in
    doubles (Table 1: sums over the vertices of their draw sequences)."""
    rp = row_ptr.cpu().numpy()
    d = np.diff(rp)
    w = (d[col.cpu().numpy()] - 1).astype(np.int64)
    pad = np.concatenate([[0], np.cumsum(w)])
    S = pad[rp[1:]] - pad[rp[:-1]]
    del pad

    # products by pieces of 24 bits, so that no sum leaves 64 bits
    def total(x, y):
        return sum(_dot(x >> i & 0xFFFFFF, y >> j & 0xFFFFFF) << (i + j) for i in (0, 24, 48) for j in (0, 24, 48))

    gamma = total(S, np.maximum(d - 1, 0))
    gamma1 = total(S, np.maximum((d - 1) * (d - 2), 0))
    gamma2 = total(S, S) - total(w, w)
    lam3 = sum((d * (d - 1) * (d - 2) // 6).tolist())
    pairs = d * (d - 1) // 2
    lam4 = sum(p * (int(x) - 2) * (int(x) - 3) // 12 for p, x in zip(pairs.tolist(), d.tolist()) if x >= 4)
    return np.array([float(gamma), float(gamma1), float(gamma2)]), float(lam3), float(lam4), int(d.max())


def _dot(x: np.ndarray, y: np.ndarray) -> int:
    """sum x y of 24-bit values, in pieces whose sums stay within 62 bits."""
    return sum(int(np.dot(x[i:i + 8192], y[i:i + 8192])) for i in range(0, len(x), 8192))


def _mix5(K, hits, gamma, lam4):
    """The MOSS-5 estimates, variances and covariances (Theorems 6-10) of
    T-5 and Path-5 counts; a class both can see is weighted by the inverse
    variances at the pooled estimate."""
    K, m = K.astype(np.float64), hits.astype(np.float64)
    p = np.zeros((2, 22))
    p[:, 1:] = 2.0 * _PHI5[:, :2].T / np.asarray(gamma)[1:, None]
    with np.errstate(divide="ignore", invalid="ignore"):
        single = np.where(p > 0, m / (K[:, None] * p), 0.0)
        both = (p > 0).all(axis=0)
        plug = np.where(both, m.sum(axis=0) / (K[:, None] * p).sum(axis=0), single.sum(axis=0))
        var = np.maximum(np.where(p > 0, plug / K[:, None] * (1.0 / p - plug), 0.0), 0.0)
        lam = np.where(both & (var.sum(axis=0) > 0), var[::-1] / var.sum(axis=0), np.where(both, 0.5, (p > 0) * 1.0))
    lam, plug = np.nan_to_num(lam), np.nan_to_num(plug)
    for a in (lam, plug):
        a[..., [0, 2]] = 0.0
    est = (lam * single).sum(axis=0)
    out_var = np.where(both, lam[0] * var[0], var.sum(axis=0))   # V1 V2 / (V1 + V2), or the one source's
    cov = -sum(np.outer(lam[l] * plug, lam[l] * plug) / K[l] for l in range(2))
    out_var[[0, 2]] = 0.0
    np.fill_diagonal(cov, out_var)
    star = np.zeros(22)
    star[1:] = _PHI5[:, 2]
    star[2] = 0.0   # class 2 is the 4-star itself: Lambda4 less the stars of the others
    est[2] = lam4 - star @ est
    cov[2, :] = cov[:, 2] = -(star @ cov)
    cov[2, 2] = out_var[2] = star @ np.where(np.outer(star, star) > 0, cov, 0.0) @ star
    return est, out_var, lam, cov


def exact(case: dict, seed: int):
    if case["do"] == "finalize":
        gamma, _, lam4, _ = _totals(*_graph(case, seed))
        K, hits = _shard_counts(case, seed)
        est, var, lam, cov = _mix5(K, hits, gamma, lam4)
        return {"cov": cov, "k": 5, "K": (int(K[0]), int(K[1])), "hits": hits, "est": est, "var": var, "lam": lam,
                "triangles": 0.0, "triangles_var": 0.0, "conc": est / est[1:].sum()}
    if case["do"] == "step" and case["n"] <= 1_100_000:
        gamma, lam3, lam4, d_max = _totals(*_graph(case, seed))
        which = {"4": ["estimate"], "5": ["estimate"], "4min": ["mix"], "all": ["mix", "estimate"]}[case["tables"]]
        return {**{w: None for w in which},
                "totals": {"gamma": gamma, "lambda3": lam3, "lambda4": lam4, "d_max": d_max}}
    return None
