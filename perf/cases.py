"""Timed workloads of the library: what a user has it do, through the public
entry points of paper_2311_00869_gb300, over the range of sizes it serves.

listed()            the fixed cases
draw(rng)           one more case of the same ranges
prepare(case, seed) inputs and the loaded context a program holds before the call
run(state)          one pass, returning every output
work(case)          bytes and operations one pass cannot do without
exact(case, seed)   the float outputs in 64 bits, without this package

Graphs are drawn on the GPU from the seed alone: R-MAT (0.57, 0.19, 0.19, 0.05)
with two planted factions (equal, 10 % sign noise) or three (94.8 / 2.6 / 2.6 %,
15 % noise), Erdos-Renyi with 20 % negative edges, and batches of uneven
Chung-Lu graphs (exponent 2.5, mean degree 8, vertex counts log-uniform).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2311_00869_gb300 as P

DEV = "cuda"


# ------------------------------------------------------------------ the cases
# ids an R-MAT graph is drawn over, vertices of its largest component, edges
RMAT17 = {"ids": 1 << 17, "n": 95001, "m": 1 << 20}
RMAT20 = {"ids": 1 << 20, "n": 656230, "m": 16777042}
RMAT24 = {"ids": 1 << 24, "n": 7410123, "m": 134211713}


def listed():
    return [
        # one tree of a small graph: the plain, tree-at-a-time use of Algorithm 1;
        # latency and launches are all there is
        {"name": "tree_er1000", "kind": "bpp", "graph": "er", "n": 1000, "m": 5000, "K": 1, "cloud": False,
         "label": False},
        # the paper's small setting batched: 64 trees, counts and the cloud
        {"name": "bpp_er1000_K64", "kind": "bpp", "graph": "er", "n": 1000, "m": 5000, "K": 64, "cloud": True,
         "label": False},
        # a middling social network (about the size of the SNAP signed graphs) with a
        # ragged tree count, labels exported for further analysis
        {"name": "bpp_rmat17_K1000", "kind": "bpp", "graph": "rmat2", **RMAT17, "K": 1000,
         "cloud": True, "label": True},
        # the benchmark's 2^20 line: 1024 trees per step
        {"name": "bpp_rmat20_K1024", "kind": "bpp", "graph": "rmat2", **RMAT20, "K": 1024, "cloud": True,
         "label": True},
        # the benchmark's headline: 2^24 ids, 2^27 edges, 4096 trees per step
        {"name": "bpp_rmat24_K4096", "kind": "bpp", "graph": "rmat3", **RMAT24, "K": 4096,
         "cloud": True, "label": False},
        # many uneven graphs in one union, whole steps without host synchronisation
        {"name": "batch_512x256", "kind": "batch", "graph": "chunglu", "graphs": 512, "n_lo": 50, "n_hi": 50000,
         "K": 256, "steps": 3},
        # the other tree sampler
        {"name": "kruskal_rmat20_K256", "kind": "kruskal", "graph": "rmat2", **RMAT20, "K": 256},
        # graphL inside a training program: loss and its gradient through autograd
        {"name": "loss_rmat20_R64", "kind": "loss", "graph": "rmat2", **RMAT20, "R": 64},
        # graphL descent as the benchmark runs it: 256 start points, 128-column segments
        # (the tuned width), the discrete loss traced
        {"name": "descent_rmat20_R256", "kind": "descent", "graph": "rmat2", **RMAT20, "R": 256,
         "steps": 25, "alpha": 0.05, "trace": True, "lanes": 32},
        # graphL on a small graph with a few restarts, default knobs: odd width, many short steps
        {"name": "descent_er1000_R5", "kind": "descent", "graph": "er", "n": 1000, "m": 5000, "R": 5, "steps": 100,
         "alpha": 0.05, "trace": False, "lanes": 0},
        # Algorithm 2's final loop: losses of given points and the edges each one flips
        {"name": "round_rmat17_R96", "kind": "round", "graph": "rmat2", **RMAT17, "R": 96},
        # a graph arriving from pinned host memory: cleaning, component, CSR
        {"name": "ingest_rmat20", "kind": "ingest", "graph": "rmat2", **RMAT20},
    ]


def _log_int(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))


def draw(rng):
    kind = rng.choice(["bpp", "bpp", "bpp", "batch", "kruskal", "loss", "descent", "descent", "round", "ingest"])
    if kind == "batch":
        hi = _log_int(rng, 500, 50000)
        graphs = _log_int(rng, 8, min(2048, int(4e6 / (hi / 6))))
        return {"kind": "batch", "graph": "chunglu", "graphs": graphs, "n_lo": 50, "n_hi": hi,
                "K": _log_int(rng, 1, 256), "steps": rng.randint(1, 4)}
    graph = rng.choice(["er", "rmat2", "rmat2", "rmat3"])
    n = _log_int(rng, 500, 1 << (21 if kind == "bpp" else 20))
    case = {"kind": kind, "graph": graph}
    if graph == "er":
        case.update(n=n, m=int(n * rng.uniform(4, 6)))
    else:  # the smaller the graph, the fewer ids the edges miss
        case.update(ids=n, n=int(n * (1 - 0.018 * math.log2(n))), m=int(n * rng.uniform(8, 16)))
    m = case["m"]
    if kind == "bpp":
        case.update(K=_log_int(rng, 1, max(1, min(4096, int(2.5e10 / m)))), cloud=rng.random() < 0.7,
                    label=rng.random() < 0.4)
    elif kind == "kruskal":
        case.update(K=_log_int(rng, 1, max(1, min(1024, int(4e9 / m)))))
    elif kind in ("loss", "round"):
        case.update(R=_log_int(rng, 1, 256))
    elif kind == "descent":
        case.update(R=_log_int(rng, 1, 256), steps=_log_int(rng, 5, 50), alpha=0.05, trace=rng.random() < 0.5,
                    lanes=rng.choice([0, 0, 16, 32]))
    return case


# ------------------------------------------------------------------ the inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _component(n, u, v):
    """Mask of the largest connected component's vertices."""
    root = torch.arange(n, device=DEV)
    while True:
        low = root.clone()
        low.scatter_reduce_(0, u, root[v], "amin")
        low.scatter_reduce_(0, v, root[u], "amin")
        low = low[low]
        if torch.equal(low, root):
            return root == torch.bincount(root, minlength=n).argmax()
        root = low


def _pairs(case, gen):
    """Distinct pairs (keys lo * ids + hi) in random order, a few per cent more
    than the case's edges."""
    ids, m = case.get("ids", case["n"]), case["m"]
    keys = torch.zeros(0, dtype=torch.int64, device=DEV)
    want = int(m * 1.04) + 64
    while keys.numel() < want:
        k = int((want - keys.numel()) * 1.12) + 64
        if case["graph"] == "er":
            a, b = (torch.randint(0, ids, (k,), device=DEV, generator=gen) for _ in range(2))
        else:
            scale = max(1, (ids - 1).bit_length())
            a = torch.zeros(k, dtype=torch.int64, device=DEV)
            b = torch.zeros(k, dtype=torch.int64, device=DEV)
            for _ in range(scale):
                r = torch.rand(k, device=DEV, generator=gen)
                a = a * 2 + (r >= 0.76)
                b = b * 2 + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
            a, b = a * ids >> scale, b * ids >> scale
        lo, hi = torch.minimum(a, b), torch.maximum(a, b)
        keys = torch.unique(torch.cat([keys, (lo * ids + hi)[lo != hi]]))
    return keys[torch.randperm(keys.numel(), device=DEV, generator=gen)]


def _graph(case, seed):
    """(n, src int32, dst int32, sign int8) on the GPU: a connected graph of
    exactly n vertices and m distinct edges.  It is the largest component of
    the drawn pairs, less some leaves or with stray vertices joined to a random
    edge's end until n are left, filled up to m edges with further pairs."""
    gen = _gen(seed)
    ids, n, m = case.get("ids", case["n"]), case["n"], case["m"]
    keys = _pairs(case, gen)
    u, v = keys[: m - n] // ids, keys[: m - n] % ids
    keep = _component(ids, u, v)
    inside = keep[u]
    u, v = u[inside], v[inside]
    extra = int(keep.sum()) - n
    if extra > 0:  # take leaves off (R-MAT components have many)
        deg = torch.bincount(torch.cat([u, v]), minlength=ids)
        leaves = torch.nonzero(keep & (deg == 1)).flatten()
        keep[leaves[torch.randperm(leaves.numel(), device=DEV, generator=gen)[:extra]]] = False
        inside = keep[u] & keep[v]
        u, v = u[inside], v[inside]
    elif extra < 0:
        stray = torch.nonzero(~keep).flatten()
        stray = stray[torch.randperm(stray.numel(), device=DEV, generator=gen)[:-extra]]
        u = torch.cat([u, u[torch.randint(0, u.numel(), (-extra,), device=DEV, generator=gen)]])
        v = torch.cat([v, stray])
        keep[stray] = True
    more = keys[m - n:]
    more = more[keep[more // ids] & keep[more % ids]]
    more = more[~torch.isin(more, torch.minimum(u, v)[-n:] * ids + torch.maximum(u, v)[-n:])]
    more = more[: m - u.numel()]
    u, v = torch.cat([u, more // ids]), torch.cat([v, more % ids])
    name = torch.full((ids,), -1, device=DEV)
    name[keep] = torch.randperm(n, device=DEV, generator=gen)
    u, v = name[u], name[v]
    turn = torch.rand(m, device=DEV, generator=gen) < 0.5
    u, v = torch.where(turn, v, u), torch.where(turn, u, v)
    x = torch.rand(n, device=DEV, generator=gen)
    if case["graph"] == "er":
        fac, noise = torch.zeros_like(x), 0.20
    elif case["graph"] == "rmat2":
        fac, noise = (x < 0.5).int(), 0.10
    else:
        fac, noise = (x >= 0.948).int() + (x >= 0.974).int(), 0.15
    sign = torch.where(fac[u] == fac[v], 1, -1)
    sign = torch.where(torch.rand(m, device=DEV, generator=gen) < noise, -sign, sign)
    return n, u.int(), v.int(), sign.to(torch.int8)


def _uncleaned(n, u, v, s, seed):
    """The graph as a file would hold it: one edge in 50 listed again the other
    way round, and one vertex in 50 outside the large component."""
    gen = _gen(seed + 2)
    again = torch.randint(0, u.numel(), (u.numel() // 50,), device=DEV, generator=gen)
    stray = n + torch.arange(2 * (n // 100), device=DEV, dtype=torch.int32)
    parts = [torch.cat([u, v[again], stray[::2]]), torch.cat([v, u[again], stray[1::2]]),
             torch.cat([s, s[again], s.new_ones(n // 100)])]
    order = torch.randperm(parts[0].numel(), device=DEV, generator=gen)
    return (n + stray.numel(), *(p[order].cpu().pin_memory() for p in parts))


def _batch_graphs(case, seed):
    """List of (n, src, dst, sign) numpy graphs: uneven Chung-Lu."""
    gen = _gen(seed)
    G = case["graphs"]
    x = torch.rand(G, device=DEV, generator=gen, dtype=torch.float64)
    nv = (case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** x).long()
    voff = torch.cat([nv.new_zeros(1), nv.cumsum(0)])
    gid = torch.repeat_interleave(torch.arange(G, device=DEV), (nv * 4.6).long())
    N = int(voff[-1])

    def endpoint():  # weights (i + 1)^(-2/3): i = n u^3
        r = torch.rand(gid.numel(), device=DEV, generator=gen, dtype=torch.float64)
        return voff[gid] + torch.minimum((nv[gid] * r ** 3).long(), nv[gid] - 1)

    a, b = endpoint(), endpoint()
    lo, hi = torch.minimum(a, b), torch.maximum(a, b)
    key = torch.unique((lo * N + hi)[lo != hi])
    vg = torch.repeat_interleave(torch.arange(G, device=DEV), nv)
    # random order of the vertices inside each graph
    place = torch.empty(N, dtype=torch.int64, device=DEV)
    place[torch.argsort(vg + torch.rand(N, device=DEV, generator=gen, dtype=torch.float64))] = torch.arange(N, device=DEV)
    g = vg[key // N]
    u, v = place[key // N] - voff[g], place[key % N] - voff[g]
    neg = 0.05 + 0.25 * torch.rand(G, device=DEV, generator=gen)
    sign = torch.where(torch.rand(u.numel(), device=DEV, generator=gen) < neg[g], -1, 1)
    cut = torch.bincount(g, minlength=G).cumsum(0)[:-1].cpu().numpy()
    parts = [np.split(t.cpu().numpy(), cut) for t in (u.int(), v.int(), sign.to(torch.int8))]
    return [(int(n), s, d, w) for n, s, d, w in zip(nv.tolist(), *parts)]


def _gamma(n, R, seed):
    """graphL start points, U(-1, 1)."""
    return torch.rand((n, R), device=DEV, generator=_gen(seed + 1)) * 2 - 1


def prepare(case, seed):
    sb = P.SignedBal(0)
    st = {"case": case, "sb": sb, "seed": seed & 0xFFFF}
    if case["kind"] == "batch":
        sb.load_batch(_batch_graphs(case, seed))
        return st
    n, u, v, s = _graph(case, seed)
    if case["kind"] == "ingest":
        st["coo"] = _uncleaned(n, u, v, s, seed)
        return st
    sb.load_graph(n, u, v, s)
    del u, v, s
    if "R" in case:
        st["gamma"] = _gamma(sb.n, case["R"], seed)
        if case["kind"] == "loss":
            st["gamma"].requires_grad_()
        if case.get("lanes"):
            sb.set_tuning(gl_lanes=case["lanes"])
    return st


# ------------------------------------------------------------------ one pass
def run(st):
    case, sb = st["case"], st["sb"]
    kind = case["kind"]
    if kind == "bpp":
        if case["cloud"]:
            sb.cloud_reset()  # this pass's own cloud
        sb.sample_trees(st["seed"], 0, case["K"])
        counts, hashes = sb.frustration()
        out = [counts, hashes]
        if case["cloud"]:
            entries, fr_min = sb.cloud()
            out += [entries["hash"], entries["S"], entries["count"], entries["first_tree"], fr_min]
        if case["label"]:
            out.append(sb.label())
        return out
    if kind == "batch":
        fr_min, n_states = sb.batch_steps(st["seed"], 0, case["K"], case["steps"])
        counts, hashes = sb.frustration()  # of the last step's trees
        return [fr_min, n_states, counts, hashes]
    if kind == "kruskal":
        sb.sample_trees_kruskal(st["seed"], 0, case["K"])
        return [*sb.frustration(), sb.label()]
    if kind == "loss":
        gamma = st["gamma"]
        gamma.grad = None
        loss = P.GraphLLoss.apply(gamma, sb)
        loss.sum().backward()
        return [loss.detach(), gamma.grad]
    if kind == "descent":
        out, exps, trace, final = sb.graphL_descent(st["gamma"], case["alpha"], case["steps"], trace=case["trace"])
        return [out, exps, final] + ([trace] if case["trace"] else [])
    if kind == "round":
        loss, F = sb.graphL_fwd(st["gamma"])
        F2, flip = sb.graphL_round(st["gamma"], want_flip=True)
        return [loss, F, F2, flip]
    if kind == "ingest":
        n1, m1, _ = sb.load_graph(*st["coo"])
        return [n1, m1, *sb.graph_csr()]
    raise ValueError(kind)


# ------------------------------------------------------------------ its work
def work(case):
    """An operation is one edge of one tree, or of one column's sum."""
    kind = case["kind"]
    if kind == "batch":
        n = case["graphs"] * (case["n_hi"] - case["n_lo"]) / math.log(case["n_hi"] / case["n_lo"])
        m, K = 4 * n, case["K"] * case["steps"]
        return {"bytes": 8 * m + 4 * n + n * K / 8 + 12 * case["graphs"] * case["K"], "flops": K * m}
    m = case["m"]
    n = case["n"]
    graph = 8 * m + 4 * n  # CSR, each edge from both ends
    if kind in ("bpp", "kruskal"):
        K = case["K"]
        return {"bytes": graph + 8 * n * math.ceil(K / 64) + 12 * K, "flops": K * m}
    if kind == "ingest":
        return {"bytes": 9 * m + graph + 2 * m, "flops": 0}
    R = case["R"]
    gamma = 4 * n * R
    if kind == "loss":
        return {"bytes": 2 * graph + 3 * gamma, "flops": 4 * m * R + 4 * m * R}
    if kind == "descent":
        return {"bytes": case["steps"] * (graph + 2 * gamma), "flops": case["steps"] * 4 * m * R}
    if kind == "round":
        return {"bytes": 8 * m + gamma + m * R / 8 + 12 * R, "flops": 4 * m * R}
    raise ValueError(kind)


# ------------------------------------------------------------------ 64 bits
def _exact_adjacency(case, seed):
    """Signed adjacency matrix in 64 bits."""
    n, u, v, s = _graph(case, seed)
    u, v, s = u.long(), v.long(), s.double()
    A = torch.sparse_coo_tensor(torch.stack([torch.cat([u, v]), torch.cat([v, u])]), torch.cat([s, s]), (n, n))
    return A.coalesce().to_sparse_csr()


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("loss", "descent", "round"):
        return None  # whole numbers only
    A = _exact_adjacency(case, seed)
    m = case["m"]
    G = _gamma(case["n"], case["R"], seed).double()
    if kind in ("loss", "round"):
        AG = A @ G
        loss = 0.5 * m - 0.25 * (G * AG).sum(0)
        return [loss, -0.5 * AG] if kind == "loss" else [loss, None, None, None]
    scale = torch.ones(case["R"], dtype=torch.float64, device=DEV)
    for _ in range(case["steps"]):
        G = G * scale
        G = G + 0.5 * case["alpha"] * (A @ G)
        scale = torch.where(G.abs().amax(0) >= 2.0 ** 32, 2.0 ** -32, 1.0).double()
    return [G * scale, None, None] + ([None] if case["trace"] else [])
