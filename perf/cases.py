"""The workloads that this library's speed is measured on.

Each case is one call, or a short fixed sequence of calls, of the public Python
binding, as a program that uses the library makes it: the graph is loaded once
and its handle kept, then the call is made on it.  ``listed`` gives the fixed
cases, ``draw`` more of the same ranges, ``prepare`` the state of a case from a
seed, ``run`` one pass, ``work`` the bytes and operations that a pass cannot do
without, and ``exact`` the same results from the definitions, where that is
quick.

Graph families (all connected, simple, undirected):
  ba    preferential attachment, n vertices, m edges per new vertex
  rmat  R-MAT, 2**scale ids, edge_factor * 2**scale sampled pairs, largest
        component (drawn on the GPU: a scale-24 graph takes about a minute on
        the host)
  road  side x side grid with deleted edges and a few diagonals
"""
import math

import numpy as np
import torch

from paper_1710_01144_gb300 import gc, graphgen

DENSE_N = 4200  # largest graph whose full distance matrix ``exact`` builds


def listed():
    return [
        # the smallest whole solve (2000 vertices, 10 picks): launches and host round trips
        {"name": "greedy_ba_2000", "op": "greedy", "graph": "ba", "n": 2000, "m": 5, "k": 10},
        # a social network of ordinary size, a large group
        {"name": "greedy_rmat_s20", "op": "greedy", "graph": "rmat", "scale": 20, "edge_factor": 16, "k": 100},
        # the largest graph: 8.9M vertices, 0.5G adjacency entries
        {"name": "greedy_rmat_s24", "op": "greedy", "graph": "rmat", "scale": 24, "edge_factor": 16, "k": 50},
        # a road network: hundreds of BFS levels, no hubs
        {"name": "greedy_road_256", "op": "greedy", "graph": "road", "side": 256, "k": 20},
        # exact gains of a list of candidates, host arrays in and out (ragged last batch)
        {"name": "gains_rmat_s20", "op": "gains", "graph": "rmat", "scale": 20, "edge_factor": 16, "group": 10,
         "candidates": 4001},
        # the same on a deep graph, device arrays in and out (asynchronous)
        {"name": "gains_road_512", "op": "gains_device", "graph": "road", "side": 512, "group": 50,
         "candidates": 1001},
        # farness of a given group: one multi-source BFS
        {"name": "farness_rmat_s20", "op": "farness", "graph": "rmat", "scale": 20, "edge_factor": 16, "group": 100},
        # many graphs of mixed family, size and k in one call, as a serving batch
        {"name": "batch_mix_24", "op": "batch", "graph": "mix", "count": 24, "n_hi": 500000},
        # top-k closeness
        {"name": "topk_rmat_s18", "op": "topk", "graph": "rmat", "scale": 18, "edge_factor": 16, "k": 100},
        # the weighted greedy, weights in [1, 16]
        {"name": "weighted_rmat_s14", "op": "weighted", "graph": "rmat", "scale": 14, "edge_factor": 16, "k": 50},
        # bitGreedy++ on a small flat graph, where it is used
        {"name": "bits_road_64", "op": "bits", "graph": "road", "side": 64, "k": 50},
        # the proposal network: scores of a list of candidates, and a gradient of the same rows
        {"name": "mlp_16k", "op": "mlp", "rows": 16384},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case; sizes are drawn on a logarithmic scale."""
    op = rng.choice(["greedy", "greedy", "greedy", "gains", "gains_device", "farness", "batch", "topk", "weighted", "bits",
                     "mlp"])
    if op == "mlp":
        return {"op": op, "rows": _log(rng, 1, 16384)}
    if op == "batch":
        return {"op": op, "graph": "mix", "count": rng.randint(2, 24), "n_hi": _log(rng, 20000, 500000)}
    fam = rng.choice(["ba", "rmat", "rmat", "road"])
    c = {"op": op, "graph": fam}
    if fam == "ba":
        c["n"] = _log(rng, 500, {"weighted": 8000, "bits": 8000, "topk": 60000}.get(op, 200000))
        c["m"] = rng.randint(2, 12)
    elif fam == "rmat":
        c["scale"] = rng.randint(9, {"greedy": 23, "topk": 18, "weighted": 14, "bits": 12}.get(op, 22))
        c["edge_factor"] = rng.randint(6, 16)
    else:
        c["side"] = _log(rng, 20, {"greedy": 220, "topk": 128, "weighted": 64, "bits": 64}.get(op, 512))
    if op in ("greedy", "topk", "weighted", "bits"):
        c["k"] = _log(rng, 3, 50 if op in ("weighted", "bits") else 100)
    else:
        c["group"] = _log(rng, 1, 100)
        if op != "farness":
            c["candidates"] = min(_log(rng, 1, 1500 if fam == "road" else 8000), _entries(c)[0] // 2)
    return c


# ------------------------------------------------------------------ inputs --
def _rmat(scale, edge_factor, seed):
    """R-MAT CSR (a, b, c = .57, .19, .19) as int32 CUDA tensors: symmetrised,
    deduplicated, no self-loops, the component of the largest degree, ids kept
    in order."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    pairs, step = edge_factor << scale, 1 << 24
    n = 1 << scale
    parts = []
    for lo in range(0, pairs, step):
        cnt = min(step, pairs - lo)
        u = torch.zeros(cnt, dtype=torch.int64, device="cuda")
        v = torch.zeros(cnt, dtype=torch.int64, device="cuda")
        for _ in range(scale):
            r = torch.rand(cnt, device="cuda", generator=g)
            down = r >= 0.76
            right = ((r >= 0.57) & (r < 0.76)) | (r >= 0.95)
            u = u * 2 + down
            v = v * 2 + right
        keep = u != v
        u, v = u[keep], v[keep]
        parts.append(torch.unique(torch.cat([(u << scale) | v, (v << scale) | u])))
    key = torch.unique(torch.cat(parts)) if len(parts) > 1 else parts[0]
    del parts
    src, dst = key >> scale, key & (n - 1)
    del key
    deg = torch.bincount(src, minlength=n)
    seen = torch.zeros(n, dtype=torch.bool, device="cuda")
    seen[deg.argmax()] = True
    count = 1
    while True:
        seen[dst[seen[src]]] = True
        now = int(seen.sum())
        if now == count:
            break
        count = now
    new_id = torch.cumsum(seen, 0) - 1
    if count < n:
        keep = seen[src]
        src, dst = src[keep], dst[keep]
    rp = torch.zeros(count + 1, dtype=torch.int32, device="cuda")
    rp[1:] = torch.cumsum(deg[seen], 0)
    ci = new_id[dst].to(torch.int32)
    return rp, ci


def _graph(case, seed):
    """(row_ptr, col_idx): CUDA tensors for rmat, numpy arrays otherwise."""
    if case["graph"] == "rmat":
        return _rmat(case["scale"], case["edge_factor"], seed)
    if case["graph"] == "ba":
        return graphgen.barabasi_albert(case["n"], case["m"], seed + 1)
    return graphgen.grid_road(case["side"], case["side"], 0.2, 0.01, seed + 1)


def _host(rp, ci):
    if torch.is_tensor(rp):
        return rp.cpu().numpy(), ci.cpu().numpy()
    return rp, ci


def _group_and_candidates(case, rp, seed):
    """A group as greedy picks them (hubs on graphs that have them, else
    anywhere) and distinct candidates from the whole graph."""
    rp = rp.cpu().numpy() if torch.is_tensor(rp) else rp
    n = rp.size - 1
    rng = np.random.default_rng(seed)
    s = min(case["group"], n)
    if case["graph"] == "road":
        S = rng.choice(n, s, replace=False)
    else:
        S = np.argsort(-np.diff(rp), kind="stable")[:s]
    c = min(case.get("candidates", 0), n)
    cand = rng.choice(n, c, replace=False)
    return S.astype(np.int32), cand.astype(np.int32)


def _mix(case, seed):
    """The mixed batch's families, sizes and k, the graphs themselves by seed."""
    items = graphgen.batch_params(case["count"], seed=1, n_hi=case["n_hi"])
    for i in items:
        i.seed = (i.seed + 0x9E3779B97F4A7C15 * seed) % (1 << 63)
    return [graphgen.batch_graph(i) for i in items], [i.k for i in items]


def _mlp_inputs(case, seed):
    """Parameters as the proposal's training starts from, rows with the ranges
    of the eight features and log-gain targets."""
    rng = np.random.default_rng(seed)
    sizes = [((8, 64), 8), ((64,), 0), ((64, 64), 64), ((64,), 0), ((64,), 64), ((1,), 0)]
    p = np.concatenate([rng.normal(0, math.sqrt(2.0 / f), s).ravel() if f else np.zeros(s) for s, f in sizes])
    m = case["rows"]
    ub = rng.uniform(0, 14, m)
    X = np.stack([rng.uniform(0.7, 9, m), rng.integers(1, 6, m), ub, rng.integers(0, 50, m), rng.uniform(2, 16, m),
                  rng.integers(0, 3, m), np.full(m, rng.uniform(4, 12)), ub], axis=1)
    X[:, 7] -= X[:, 6]
    y = np.maximum(0.0, ub - rng.exponential(1.0, m))
    return p.astype(np.float32), X.astype(np.float32), y.astype(np.float32)


def prepare(case, seed):
    op = case["op"]
    if op == "mlp":
        p, X, y = _mlp_inputs(case, seed)
        net = gc.Mlp(max_batch=max(1, case["rows"]))
        net.set_params(p)
        return {"op": op, "net": net, "X": torch.from_numpy(X).cuda(), "y": torch.from_numpy(y).cuda(),
                "out": torch.empty(case["rows"], dtype=torch.float32, device="cuda")}
    if op == "batch":
        graphs, ks = _mix(case, seed)
        return {"op": op, "batch": gc.Batch(graphs), "ks": ks}
    rp, ci = _graph(case, seed)
    st = {"op": op, "G": gc.Graph(rp, ci), "k": case.get("k")}
    if op in ("gains", "gains_device", "farness"):
        st["S"], st["cand"] = _group_and_candidates(case, rp, seed)
    if op == "gains_device":
        st["S"], st["cand"] = torch.from_numpy(st["S"]).cuda(), torch.from_numpy(st["cand"]).cuda()
        st["out"] = torch.empty(st["cand"].numel(), dtype=torch.int64, device="cuda")
    if op == "weighted":
        st["G"].set_weights(graphgen.edge_weights(*_host(rp, ci), 16, seed + 1))
    return st


# -------------------------------------------------------------------- calls --
def run(state):
    op = state["op"]
    if op == "greedy":
        group, farness, _ = state["G"].greedy(state["k"])
        return {"group": group, "farness": farness}
    if op == "gains":
        return {"gains": state["G"].gains(state["S"], state["cand"])}
    if op == "gains_device":
        state["G"].gains_device(state["S"], state["cand"], state["out"])
        return {"gains": state["out"]}
    if op == "farness":
        return {"farness": state["G"].farness(state["S"])}
    if op == "batch":
        groups, farness, _ = state["batch"].greedy(state["ks"])
        return {"groups": np.concatenate(groups), "farness": farness}
    if op == "topk":
        ids, farness, _ = state["G"].top_closeness(state["k"])
        return {"ids": ids, "farness": farness}
    if op == "weighted":
        group, farness, _ = state["G"].greedy_weighted(state["k"])
        return {"group": group, "farness": farness}
    if op == "bits":
        group, farness, _ = state["G"].greedy_bits(state["k"])
        return {"group": group, "farness": farness}
    state["net"].forward(state["X"], state["out"])
    grad, loss = state["net"].grad(state["X"], state["y"])
    return {"out": state["out"], "grad": grad, "loss": np.float32(loss)}  # the loss of float32 outputs


def _entries(case):
    """About how many vertices and adjacency entries the case's graph has."""
    if case["graph"] == "ba":
        return case["n"], 2 * case["n"] * case["m"]
    if case["graph"] == "rmat":  # isolated ids and repeated pairs drop out
        return int(0.57 * 2 ** case["scale"]), int(1.93 * case["edge_factor"] * 2 ** case["scale"])
    return int(0.995 * case["side"] ** 2), int(3.24 * case["side"] ** 2)


def work(case):
    """Graph cases: the CSR (and weights) read once, the outputs written once.
    The proposal network: its rows and parameters read once; multiply-adds of
    one forward pass for the scores and one forward and backward pass."""
    op = case["op"]
    if op == "mlp":
        m = case["rows"]
        macs = 8 * 64 + 64 * 64 + 64
        return {"bytes": 4.0 * (m * 10 + 2 * 4801), "flops": 2.0 * m * (2 * macs + macs + 64 * 64 + 64)}
    if op == "batch":
        n = e = k = 0
        for i in graphgen.batch_params(case["count"], seed=1, n_hi=case["n_hi"]):
            n, e, k = n + i.n_target, e + int(i.n_target * i.avg_deg), k + i.k
        return {"bytes": 4.0 * (n + e + k) + 8.0 * case["count"], "flops": 0}
    n, e = _entries(case)
    out = {"gains": 12, "gains_device": 12}.get(op, 0) * case.get("candidates", 0) + 12 * case.get("k", 0) \
        + 4 * case.get("group", 0) + 8
    return {"bytes": 4.0 * n + (8.0 if op == "weighted" else 4.0) * e + out, "flops": 0}


# ------------------------------------------------- results by definition --
def _dense_distances(rp, ci, w=None):
    """int64 distance matrix on the GPU."""
    n = rp.size - 1
    src = torch.from_numpy(np.repeat(np.arange(n), np.diff(rp))).cuda()
    dst = torch.from_numpy(ci.astype(np.int64)).cuda()
    if w is not None:
        D = torch.full((n, n), 1 << 40, dtype=torch.int64, device="cuda")
        D[src, dst] = torch.from_numpy(w.astype(np.int64)).cuda()
        D.fill_diagonal_(0)
        for v in range(n):
            torch.minimum(D, D[:, v:v + 1] + D[v:v + 1, :], out=D)
        return D
    A = torch.zeros((n, n), dtype=torch.float32, device="cuda")
    A[src, dst] = 1
    seen = torch.eye(n, dtype=torch.bool, device="cuda")
    D = torch.zeros((n, n), dtype=torch.int64, device="cuda")
    front, level = seen.float(), 0
    while True:
        new = ((A @ front) > 0) & ~seen
        level += 1
        if not bool(new.any()):
            return D
        D[new] = level
        seen |= new
        front = new.float()


def _first_best(x):
    return int(np.argmax(x.cpu().numpy()))  # the smallest id among equals


def _greedy_exact(D, k):
    group = [_first_best(-D.sum(1))]
    dS = D[group[0]].clone()
    for _ in range(k - 1):
        gain = (dS[None, :] - D).clamp(min=0).sum(1)
        gain[group] = -1
        group.append(_first_best(gain))
        dS = torch.minimum(dS, D[group[-1]])
    return {"group": np.array(group, dtype=np.int32), "farness": int(dS.sum())}


def _bfs_farness(rp, ci, S):
    rp, ci = torch.as_tensor(rp).cuda(), torch.as_tensor(ci).cuda().long()
    n = rp.numel() - 1
    src = torch.repeat_interleave(torch.arange(n, device="cuda"), (rp[1:] - rp[:-1]).long())
    seen = torch.zeros(n, dtype=torch.bool, device="cuda")
    seen[torch.from_numpy(S.astype(np.int64)).cuda()] = True
    total, level, count = 0, 0, int(seen.sum())
    while count < n:
        seen[ci[seen[src]]] = True
        level += 1
        now = int(seen.sum())
        total, count = total + level * (now - count), now
    return total


def exact(case, seed):
    op = case["op"]
    if op == "mlp":
        p, X, y = (torch.from_numpy(a).double() for a in _mlp_inputs(case, seed))
        p.requires_grad_(True)
        W1, b1, W2, b2, W3, b3 = torch.split(p, [512, 64, 4096, 64, 64, 1])
        h = torch.relu(X @ W1.view(8, 64) + b1)
        out = torch.relu(h @ W2.view(64, 64) + b2) @ W3 + b3
        loss = ((out - y) ** 2).mean()
        loss.backward()
        return {"out": out.detach(), "grad": p.grad, "loss": loss.detach()}
    if op == "batch":
        return None
    rp, ci = _graph(case, seed)
    if op == "farness":
        S, _ = _group_and_candidates(case, rp, seed)
        return {"farness": _bfs_farness(rp, ci, S)}
    rp, ci = _host(rp, ci)
    if rp.size - 1 > DENSE_N:
        return None
    D = _dense_distances(rp, ci, graphgen.edge_weights(rp, ci, 16, seed + 1) if op == "weighted" else None)
    if op in ("greedy", "weighted", "bits"):
        return _greedy_exact(D, min(case["k"], rp.size - 1))
    if op == "topk":
        f = D.sum(1).cpu().numpy()
        ids = np.lexsort((np.arange(f.size), f))[:case["k"]]
        return {"ids": ids.astype(np.int32), "farness": f[ids]}
    S, cand = _group_and_candidates(case, rp, seed)
    dS = D[torch.from_numpy(S.astype(np.int64)).cuda()].min(0).values
    gain = (dS[None, :] - D[torch.from_numpy(cand.astype(np.int64)).cuda()]).clamp(min=0).sum(1)
    return {"gains": gain}
