"""The work a user of this library has it do, as measurable cases.

Every case is one call of the package's public API on one seeded synthetic
graph (graphgen), with the graph where such a program has it: resident on the
GPU, or in host arrays.  Graph families, with the sizes of the repository's
workloads, tests and benchmark:

  social        config(1): a Chung-Lu core plus pendants, a few thousand vertices
  articulation  config(2): Erdos-Renyi blocks glued at cut vertices, plus chains
  side          articulation plus vertices whose neighbourhoods are cliques
  twins         config(3): a power-law core, groups of identical vertices, pendants
  unequal       a power-law core whose twins carry pendants (classes of unequal reach)
  road          config(4): a thinned grid with trees on its perimeter
  batch         many independent Chung-Lu graphs packed in one CSR
"""
import math

import numpy as np
import torch

import graphgen as gg
import paper_1209_6007_gb300 as bcs


def listed():
    return [
        # a small social graph from a notebook or a service: all latency
        {"name": "social-2.6k", "family": "social", "size": 100, "call": "shattered"},
        # the same graph in a loop that must not enter the allocator
        {"name": "social-2.6k-noalloc", "family": "social", "size": 100, "call": "noalloc"},
        # plain Brandes on a graph of ragged size, as a check on the shattered call
        {"name": "unequal-7k-plain", "family": "unequal", "size": 3511, "call": "plain"},
        # a graph that lives in host arrays, and whose result is wanted there
        {"name": "articulation-38k-host", "family": "articulation", "size": 5, "call": "shattered", "host": True},
        # the articulation workload at full size: thousands of pieces, all small
        {"name": "articulation-648k", "family": "articulation", "size": 100, "call": "shattered"},
        # vertices in many triangles (collaboration graphs): the side-vertex step
        {"name": "side-174k", "family": "side", "size": 20, "call": "shattered", "side": True},
        # twins of unequal reach merged too: one piece of some 13,000 vertices
        {"name": "unequal-25k", "family": "unequal", "size": 12500, "call": "shattered", "unequal": True},
        # the twin workload (the benchmark's headline) at a fifth of its size, FP32 dependencies
        {"name": "twins-194k-fp32", "family": "twins", "size": 20, "call": "shattered", "fp32": True},
        # scores estimated from sampled sources on a large social graph
        {"name": "twins-291k-sampled", "family": "twins", "size": 30, "call": "sources", "sources": 1000},
        # the same on a large road network, FP32 dependencies (deep searches)
        {"name": "road-683k-sampled-fp32", "family": "road", "size": 30, "call": "sources", "sources": 456, "fp32": True},
        # a town's road network, all sources
        {"name": "road-25k", "family": "road", "size": 1, "call": "shattered"},
        # a data set of independent graphs of uneven size, scored in one call
        {"name": "batch-1000-to-4096", "family": "batch", "size": 1000, "n_max": 4096, "call": "batch"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    f = rng.choice(["social", "articulation", "side", "twins", "unequal", "road", "batch"])
    fp32 = rng.random() < 0.4
    if f == "social":
        call = rng.choice(["shattered", "plain", "noalloc"])
        return {"family": f, "size": _log(rng, 10, 300), "call": call, "fp32": fp32, "host": call != "noalloc" and rng.random() < 0.3}
    if f == "articulation":
        return {"family": f, "size": _log(rng, 2, 100), "call": "shattered", "fp32": fp32, "host": rng.random() < 0.3}
    if f == "side":
        return {"family": f, "size": _log(rng, 2, 30), "call": "shattered", "fp32": fp32, "side": rng.random() < 0.7}
    if f == "twins":
        if rng.random() < 0.5:
            return {"family": f, "size": _log(rng, 2, 15), "call": "shattered", "fp32": fp32}
        return {"family": f, "size": _log(rng, 5, 30), "call": "sources", "sources": _log(rng, 64, 1500), "fp32": fp32}
    if f == "unequal":
        call = rng.choice(["shattered", "shattered", "plain"])
        return {"family": f, "size": _log(rng, 1000, 14000 if call == "shattered" else 6000), "call": call, "fp32": fp32,
                "unequal": call == "shattered" and rng.random() < 0.5}
    if f == "road":
        if rng.random() < 0.5:
            return {"family": f, "size": 1, "call": "shattered", "fp32": fp32, "cut": _log(rng, 100, 160)}
        return {"family": f, "size": _log(rng, 3, 40), "call": "sources", "sources": _log(rng, 64, 500), "fp32": fp32}
    return {"family": f, "size": _log(rng, 20, 1500), "n_max": rng.choice([300, 1024, 2500, 4096]), "call": "batch", "fp32": fp32}


def _graph(case, seed):
    """(graph, offsets of the batch's graphs or None).  The case gives the
    structure, the seed the vertex numbering (and the sources): graphs of one
    case have the same size and are searched in another order each."""
    f, size = case["family"], case["size"]
    off = None
    if f == "batch":
        g, off = gg.batch(size, seed=0xB0C00005 + case["n_max"], n_min=16, n_max=case["n_max"])
    elif f == "unequal":  # twins of uniform core vertices, pendants on any vertex
        core = gg.chung_lu(size, 2.1, 12.0, 0xB0C00007)
        rng = np.random.default_rng(size)
        parts, n = [core.edges()], core.n
        deg = core.degrees()
        pick = rng.integers(0, core.n, int(0.3 * size))
        pick = pick[deg[pick] > 0]
        parts += [np.stack([np.full(int(deg[x]), n + i, dtype=np.int64), core.neighbors(x).astype(np.int64)], 1) for i, x in enumerate(pick)]
        n += pick.size
        pend = int(0.7 * size)
        parts.append(np.stack([rng.integers(0, n, pend), np.arange(n, n + pend)], 1))
        g = gg.from_edges(n + pend, np.concatenate(parts))
    elif f == "side":
        g = gg.config(2, scale_pct=size)
        g = gg.with_side_vertices(g, 6, int(0.23 * g.n), int(0.08 * g.n))
    elif f == "road" and case.get("cut"):  # a small grid of odd size, a quarter of its edges away
        e = gg.grid(case["cut"], case["cut"] + 7).edges()
        g = gg.from_edges(case["cut"] * (case["cut"] + 7), e[np.random.default_rng(4).random(e.shape[0]) >= 0.25])
    else:
        g = gg.config({"social": 1, "articulation": 2, "twins": 3, "road": 4}[f], scale_pct=size)
    rng = np.random.default_rng(seed)
    if off is None:
        perm = rng.permutation(g.n)
    else:  # a graph of the batch keeps its range of ids
        perm = np.argsort(np.repeat(np.arange(off.size - 1), np.diff(off)) + rng.random(g.n))
    return gg.from_edges(g.n, perm[g.edges()]), off


def _sources(case, n, seed):
    return np.random.default_rng(seed + 17).choice(n, min(n, case["sources"]), replace=False)


def prepare(case, seed):
    g, off = _graph(case, seed)
    if case.get("host"):
        rp, col = g.row_ptr, g.col
    else:
        rp, col = torch.from_numpy(g.row_ptr).cuda(), torch.from_numpy(g.col).cuda()
    kw = {"delta_fp32": bool(case.get("fp32"))}
    for k in ("side", "unequal"):
        if case.get(k):
            kw[k] = True
    return {"case": case, "rp": rp, "col": col, "off": off, "kw": kw,
            "src": _sources(case, g.n, seed) if case["call"] == "sources" else None}


def run(state):
    call, rp, col, kw = state["case"]["call"], state["rp"], state["col"], state["kw"]
    if call == "plain":
        bc = bcs.bc_plain(rp, col, **kw)
    elif call == "noalloc":
        bc = bcs.bc_plain_noalloc(rp, col, **kw)
    elif call == "sources":
        bc = bcs.bc_sources(rp, col, state["src"], **kw)
    elif call == "batch":
        bc = bcs.bc_shattered_batch(state["off"], rp, col, **kw)
    else:
        bc = bcs.bc_shattered(rp, col, **kw)
    if not kw["delta_fp32"]:
        return bc
    # scores with FP32 dependencies carry FP32 accuracy: their user keeps them in FP32
    return bc.astype(np.float32) if isinstance(bc, np.ndarray) else bc.to(torch.float32)


# What Bc-Reach has to search once a graph is shattered (measured on each
# family): the square root of its (source, vertex) pairs over the input's
# vertices, and the pieces' entries per vertex.
_LEFT = {"social": (0.53, 5.1), "twins": (0.447, 13.2), "unequal": (0.55, 15.6), "road": (0.85, 3.1)}


def work(case):
    """Each input read and each output written once; per source one addition
    per shortest-path edge and direction and four operations per vertex."""
    f, size = case["family"], case["size"]
    if f == "social":
        n, deg = 26.0 * size, 3.5
    elif f in ("articulation", "side"):
        n, deg = 6476.0 * size * (1.31 if f == "side" else 1.0), 5.2
    elif f == "twins":
        n, deg = 9701.0 * size, 10.3
    elif f == "unequal":
        n, deg = 2.0 * size, 9.9
    elif f == "road":
        n, deg = (case["cut"] * (case["cut"] + 7.0), 3.0) if case.get("cut") else (22700.0 * size, 3.0)
    else:
        n, deg = size * (case["n_max"] - 16) / math.log(case["n_max"] / 16), 7.5
    nbytes = 8 * (n + 1) + 4 * n * deg + 8 * n
    if case["call"] in ("plain", "noalloc"):
        pairs = n * n
    elif case["call"] == "sources":
        pairs = case["sources"] * n
    elif f in ("articulation", "side"):
        pairs = 200.0 * n  # blocks of at most 512 vertices
    elif f == "batch":
        pairs = n * case["n_max"] / 2 * 0.7
    else:
        pairs, deg = (_LEFT[f][0] * n) ** 2, _LEFT[f][1]
    return {"bytes": nbytes, "flops": pairs * (deg + 4)}


def _brandes(rp, col, sources, column, cols):
    """Sums of the dependencies of the given sources (Brandes 2001), in FP64:
    whole levels of many searches at once as sparse-times-dense products.
    Search `column[i]` of `cols` starts at sources[i]; searches of graphs
    that share no vertex share a column."""
    n = rp.numel() - 1
    A = torch.sparse_csr_tensor(rp, col.to(torch.int64), torch.ones(col.numel(), dtype=torch.float64, device=rp.device), size=(n, n))
    bc = torch.zeros(n, dtype=torch.float64, device=rp.device)
    per = max(1, min(cols, 200_000_000 // n))
    for at in range(0, cols, per):
        mine = (column >= at) & (column < at + per)
        s, k = sources[mine], column[mine] - at
        front = torch.zeros(n, min(per, cols - at), dtype=torch.float64, device=rp.device)
        front[s, k] = 1.0
        sigma, d, level = front.clone(), torch.full(front.shape, -1, dtype=torch.int16, device=rp.device), 0
        d[s, k] = 0
        while True:
            nxt = (A @ front).masked_fill_(d >= 0, 0.0)
            new = nxt > 0
            if not bool(new.any()):
                break
            level += 1
            d[new] = level
            sigma += nxt
            front = nxt
        delta = torch.zeros_like(sigma)
        for l in range(level, 0, -1):
            c = torch.where(d == l, (1.0 + delta) / sigma.clamp(min=1.0), 0.0)
            delta += torch.where(d == l - 1, sigma * (A @ c), 0.0)
        delta[s, k] = 0.0
        bc += delta.sum(1)
    return bc


def exact(case, seed):
    g, off = _graph(case, seed)
    src = _sources(case, g.n, seed) if case["call"] == "sources" else np.arange(g.n)
    column = np.arange(src.size) if off is None else src - np.repeat(off[:-1], np.diff(off))
    cols = int(column.max()) + 1
    depth = {"road": 60 + 3.0 * math.sqrt(g.n), "articulation": 70, "side": 70}.get(case["family"], 10)
    if float(cols) * (g.nnz + 4 * g.n) * depth > 1.2e12:
        return None
    rp, col = torch.from_numpy(g.row_ptr).cuda(), torch.from_numpy(g.col).cuda()
    bc = _brandes(rp, col, torch.from_numpy(src).cuda(), torch.from_numpy(column).cuda(), cols)
    return bc.cpu().numpy() if case.get("host") else bc
