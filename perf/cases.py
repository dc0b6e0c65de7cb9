"""The work a program has this library do, as cases that can be timed.

Each case is one call (or one forward and backward pass) through the Python
binding on a graph that the program has uploaded and keeps.  The graphs are of
the two families the repository uses everywhere: "rmat" (power law, edges
sampled with quadrant probabilities .57/.19/.19/.05) and "uniform" (every edge
between two vertices drawn alike), made on the GPU from the seed alone.

listed() gives the cases, draw() further ones of the same ranges, prepare() the
graph and buffers in hand before a call, run() the call, work() the bytes and
operations one pass cannot do without, exact() the results in 64 bits by plain
torch.
"""
import math

import numpy as np
import torch

import paper_2010_16012_gb300 as gp

DEV = "cuda"
L2_BYTES = 129e6  # graphs above this are read from memory again by every sweep
MODES = {"push": gp.PUSH, "pull": gp.PULL, "auto": gp.AUTO}


def listed():
    return [
        # a small graph ranked for a fixed number of sweeps: a call of some hundred microseconds, launches count
        dict(name="rank_small", what="rank", family="rmat", n=16384, ef=16, directed=False, mode="auto", iters=20,
             tol=0.0, weighted=False, personal=False),
        # the benchmark's graph, ranked by pulling until the L1 change is below 1e-7
        dict(name="rank_pull", what="rank", family="rmat", n=4194304, ef=16, directed=False, mode="pull", iters=300,
             tol=1e-7, weighted=False, personal=False),
        # the paper's other direction: scattered updates with atomics
        dict(name="rank_push", what="rank", family="rmat", n=1000003, ef=16, directed=False, mode="push", iters=20,
             tol=0.0, weighted=False, personal=False),
        # a directed graph without skew, with a teleport vector
        dict(name="rank_uniform", what="rank", family="uniform", n=8000009, ef=16, directed=True, mode="pull", iters=20,
             tol=0.0, weighted=False, personal=True),
        # one training step through the ranks: forward and adjoint, gradients of edge weights and teleport vector
        dict(name="rank_grad", what="grad", family="rmat", n=262144, ef=16, directed=True, iters=40),
        # one search on a small graph, answered at once: latency
        dict(name="bfs_small", what="bfs", family="rmat", n=16384, ef=16, directed=False, mode="auto"),
        # the benchmark's 64 searches on its graph, levels and parents, in one call
        dict(name="bfs_many", what="bfs_multi", family="rmat", n=4194304, ef=16, directed=False, mode="auto", k=64),
        # weighted shortest paths with integer-valued weights, as in the tests
        dict(name="sssp", what="sssp", family="rmat", n=2000003, ef=16, directed=False, mode="auto", delta=64.0),
        # sampled betweenness centrality
        dict(name="bc", what="bc", family="rmat", n=1048576, ef=16, directed=False, mode="auto", k=16),
        # triangles per vertex
        dict(name="triangles", what="triangles", family="rmat", n=262144, ef=16, directed=False, mode="pull"),
        # 256 personalised ranks on each graph of a batch of unlike sizes
        dict(name="ppr_batch", what="ppr", family="rmat", n=131072, ef=16, graphs=6, k=256, tol=1e-6),
        # 64 searches on each graph of such a batch
        dict(name="msbfs_batch", what="msbfs", family="rmat", n=262144, ef=16, graphs=8, k=64),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["rank", "rank", "rank", "grad", "bfs", "bfs_multi", "sssp", "bc", "triangles", "ppr", "msbfs"])
    family = rng.choice(["rmat", "rmat", "uniform"])
    directed = rng.random() < 0.4
    ef = rng.choice([4, 8, 16, 16])
    mode = rng.choice(["auto", "auto", "pull", "push"])
    if what == "rank":
        tol = rng.choice([0.0, 0.0, 1e-7])
        return dict(what=what, family=family, n=_log_uniform(rng, 8000, 4000000), ef=ef, directed=directed, mode=mode,
                    iters=300 if tol else rng.randint(10, 30), tol=tol, weighted=rng.random() < 0.3,
                    personal=rng.random() < 0.3)
    if what == "grad":
        return dict(what=what, family=family, n=_log_uniform(rng, 8000, 500000), ef=ef, directed=True,
                    iters=rng.randint(20, 50))
    if what == "bfs":
        return dict(what=what, family=family, n=_log_uniform(rng, 8000, 4000000), ef=ef, directed=directed, mode="auto")
    if what == "bfs_multi":
        return dict(what=what, family=family, n=_log_uniform(rng, 8000, 2000000), ef=ef, directed=directed, mode="auto",
                    k=rng.randint(8, 64))
    if what == "sssp":
        return dict(what=what, family=family, n=_log_uniform(rng, 8000, 2000000), ef=ef, directed=directed, mode="auto",
                    delta=float(rng.choice([32, 64, 128])))
    if what == "bc":
        return dict(what=what, family=family, n=_log_uniform(rng, 8000, 1000000), ef=ef, directed=directed, mode="auto",
                    k=rng.randint(4, 16))
    if what == "triangles":
        return dict(what=what, family=family, n=_log_uniform(rng, 8000, 260000), ef=ef, directed=False,
                    mode=rng.choice(["pull", "push"]))
    if what == "ppr":
        return dict(what=what, family="rmat", n=_log_uniform(rng, 8000, 130000), ef=ef, graphs=rng.randint(1, 6),
                    k=rng.choice([32, 64, 128, 256]), tol=1e-6)
    return dict(what=what, family="rmat", n=_log_uniform(rng, 8000, 260000), ef=ef, graphs=rng.randint(1, 8),
                k=rng.randint(16, 64))


# ------------------------------------------------------------------ inputs


def _edges(family, n, ef, g):
    """ef * n sampled edges (source, head)."""
    count = ef * n
    if family == "uniform":
        return (torch.randint(0, n, (count,), generator=g, device=DEV),
                torch.randint(0, n, (count,), generator=g, device=DEV))
    bits = max(1, (n - 1).bit_length())
    src = torch.zeros(count, dtype=torch.int32, device=DEV)
    dst = torch.zeros(count, dtype=torch.int32, device=DEV)
    for _ in range(bits):
        r = torch.rand(count, generator=g, device=DEV)
        src.mul_(2).add_(r >= 0.76)
        dst.mul_(2).add_(((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    # any n: the 2^bits ids scaled onto it, in order
    return src.long() * n >> bits, dst.long() * n >> bits


def _compressed(rows, n):
    off = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return off


def _graph(family, n, ef, directed, g, exactly=False):
    """CSR and CSC arrays without self-loops and duplicates, rows sorted, and
    the CSR position of every CSC slot where the graph is directed.  exactly:
    ef * n edges, whatever repeats (half as many again are sampled for it)."""
    src, dst = _edges(family, n, ef + ef // 2 if exactly else ef, g)
    key = src * n + dst
    if not directed:
        key = torch.cat([key, dst * n + src])
    key = key[torch.cat([src != dst] * (1 if directed else 2))]
    key = torch.sort(key)[0]
    keep = torch.ones(key.numel(), dtype=torch.bool, device=DEV)
    keep[1:] = key[1:] != key[:-1]
    key = key[keep]
    if exactly:
        key = key[torch.sort(torch.randperm(key.numel(), generator=g, device=DEV)[:ef * n])[0]]
    src, dst = key // n, key % n
    a = {"n": n, "m": int(key.numel()), "csr_off": _compressed(src, n), "csr_idx": dst.int()}
    if directed:
        order = torch.argsort(dst, stable=True)
        a.update(csc_off=_compressed(dst, n), csc_idx=src[order].int(), perm=order)
    return a


def _sources(a, k, g):
    """k vertices with out-edges, drawn anew for every seed."""
    has = torch.nonzero(a["csr_off"][1:] > a["csr_off"][:-1]).flatten()
    pick = torch.randint(0, has.numel(), (k,), generator=g, device=DEV)
    return has[pick].int().cpu().numpy()


def _batch_sizes(case):
    """Sizes of a batch's graphs: from case["n"] down by factors of two, each a bit off."""
    return [max(1000, (case["n"] >> (i % 5)) - 37 * (i % 3)) for i in range(case["graphs"])]


def _inputs(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    what = case["what"]
    if what in ("ppr", "msbfs"):
        graphs = [_graph(case["family"], n, case["ef"], False, g) for n in _batch_sizes(case)]
        return {"graphs": graphs, "sources": np.stack([_sources(a, case["k"], g) for a in graphs])}
    a = _graph(case["family"], case["n"], case["ef"], case["directed"], g, exactly=what == "grad")
    n, m = a["n"], a["m"]
    if what == "rank":
        if case["weighted"]:  # transition weights as given: positive, normalised per source
            deg = a["csr_off"][1:] - a["csr_off"][:-1]
            row = torch.repeat_interleave(torch.arange(n, device=DEV), deg)
            w = 1.0 - torch.rand(m, generator=g, device=DEV)
            total = torch.zeros(n, dtype=torch.float64, device=DEV).index_add_(0, row, w.double())
            a["w"] = (w.double() / total[row]).float()
        if case["personal"]:
            s = torch.rand(n, generator=g, device=DEV)
            a["s"] = s / s.sum()
    elif what == "grad":
        a["w"] = 1.0 - torch.rand(m, generator=g, device=DEV)
        s = torch.rand(n, generator=g, device=DEV)
        a["s"] = s / s.sum()
        a["g"] = torch.randn(n, generator=g, device=DEV)
    elif what == "sssp":
        a["w"] = torch.randint(1, 256, (m,), generator=g, device=DEV).float()
    if what in ("bfs", "sssp", "bfs_multi", "bc"):
        a["sources"] = _sources(a, case.get("k", 1), g)
    return a


def _upload(a, **kw):
    """The graph's handle.  A directed graph, and one whose weights differ by
    direction, brings both orders."""
    if "csc_off" in a:
        w = a.get("w")
        return gp.Graph(a["n"], a["csr_off"], a["csr_idx"], a["csc_off"], a["csc_idx"], w,
                        None if w is None else w[a["perm"]], **kw)
    if "w" in a:  # undirected structure, a weight per direction: in-edge v <- u weighs what out-edge u -> v does
        return gp.Graph(a["n"], a["csr_off"], a["csr_idx"], a["csr_off"], a["csr_idx"], a["w"], a["w"][_mirror(a)], **kw)
    return gp.Graph(a["n"], a["csr_off"], a["csr_idx"], symmetric=True, **kw)


def _rows(a):
    return torch.repeat_interleave(torch.arange(a["n"], device=DEV), a["csr_off"][1:] - a["csr_off"][:-1])


def _mirror(a):
    """Undirected structure: the CSR position of the edge u -> v for every slot v <- u."""
    return torch.argsort(a["csr_idx"].long() * a["n"] + _rows(a))


def prepare(case, seed):
    a = _inputs(case, seed)
    what = case["what"]
    st = {"what": what, "case": case}
    if what in ("ppr", "msbfs"):
        graphs = [_upload(x) for x in a["graphs"]]
        st.update(graphs=graphs, sources=a["sources"], batch=gp.Batch(graphs, k_ppr=case["k"] if what == "ppr" else 32))
        return st
    if what == "grad":
        st.update(graph=_upload(a, normalize=True), perm=a["perm"], w=a["w"].requires_grad_(True),
                  s=a["s"].requires_grad_(True), g=a["g"])
        return st
    st["graph"] = _upload(a)
    if what == "rank":
        st["s"] = a.get("s")
    if "sources" in a:
        st["sources"] = a["sources"]
    if what == "bfs_multi":  # buffers that the program reuses from call to call
        st["level"] = torch.empty((case["k"], case["n"]), dtype=torch.int32, device=DEV)
        st["parent"] = torch.empty((case["k"], case["n"]), dtype=torch.int32, device=DEV)
    return st


def run(st):
    case, what = st["case"], st["what"]
    if what == "rank":
        return gp.pagerank(st["graph"], MODES[case["mode"]], 0.85, case["iters"], case["tol"],
                           personalization=st["s"])[0]
    if what == "grad":
        x = gp.pagerank_autograd(st["graph"], st["w"], st["s"], csc_perm=st["perm"], damping=0.85, iters=case["iters"],
                                 tol=0.0, adj_iters=case["iters"], adj_tol=0.0)
        gw, gs = torch.autograd.grad(x, (st["w"], st["s"]), st["g"])
        return {"ranks": x.detach(), "grad_w": gw, "grad_s": gs}
    # a search's parents are computed too, but any in-neighbour one level up may be one: two runs of one program differ
    if what == "bfs":
        return gp.bfs(st["graph"], int(st["sources"][0]), MODES[case["mode"]])[0]
    if what == "bfs_multi":
        gp.bfs_multi(st["graph"], st["sources"], MODES[case["mode"]], levels=list(st["level"]),
                     parents=list(st["parent"]))
        return st["level"]
    if what == "sssp":
        dist, pred, _ = gp.sssp(st["graph"], int(st["sources"][0]), case["delta"], MODES[case["mode"]])
        return {"dist": dist, "pred": pred}
    if what == "bc":
        return gp.bc(st["graph"], st["sources"], MODES[case["mode"]])[0]
    if what == "triangles":
        counts, total, _ = gp.triangles(st["graph"], MODES[case["mode"]])
        return {"counts": counts, "total": total}
    if what == "ppr":
        return st["batch"].ppr(st["sources"], 0.85, 1000, case["tol"])[0]
    return st["batch"].msbfs(st["sources"])[0]


# ------------------------------------------------------------------ the least work


def _m(n, ef, directed):
    """Edges of a sampled graph, about (some draws repeat or are self-loops)."""
    return 0.95 * n * ef * (1 if directed else 2)


def work(case):
    what = case["what"]
    if what in ("ppr", "msbfs"):
        sizes = [(n, _m(n, case["ef"], False)) for n in _batch_sizes(case)]
        nb = sum(4 * m + 8 * n for n, m in sizes)
        if what == "msbfs":  # the graphs read, 64 columns of levels written
            return {"bytes": nb + sum(256 * n for n, _ in sizes), "flops": 0}
        sweeps = 14  # a column's median
        return {"bytes": nb + sum(4 * n * case["k"] for n, _ in sizes),
                "flops": 2.0 * sweeps * case["k"] * sum(m for _, m in sizes)}
    n, m = case["n"], _m(case["n"], case["ef"], case["directed"])
    graph = 4 * m + 8 * n
    if what in ("rank", "grad"):
        sweeps = 20 if case.get("tol") else case["iters"]
        graph += 4 * m if what == "grad" or case["weighted"] else 0
        # a sweep reads the graph, the iterate and its scale and writes the next one; what fits in cache is read once
        reads = sweeps if graph > L2_BYTES else 1
        total = reads * (graph + 16 * n)
        if what == "grad":
            return {"bytes": 2 * total + 8 * m + 16 * n, "flops": 4.0 * m * sweeps + 4.0 * m}
        return {"bytes": total + 4 * n, "flops": 2.0 * m * sweeps}
    if what == "bfs":
        return {"bytes": graph + 8 * n, "flops": 0}
    if what == "bfs_multi":
        return {"bytes": graph + 8 * n * case["k"], "flops": 0}
    if what == "sssp":
        return {"bytes": graph + 4 * m + 8 * n, "flops": 2.0 * m}
    if what == "bc":
        reads = case["k"] if graph > L2_BYTES else 1
        return {"bytes": reads * graph + 8 * n, "flops": 4.0 * m * case["k"]}
    return {"bytes": graph + 8 * n, "flops": 0}


# ------------------------------------------------------------------ 64 bits


def _matrix(off, idx, w, n):
    return torch.sparse_csr_tensor(off, idx.long(), w, (n, n))


def _in_edges(a, w):
    """The pull matrix: row v holds P_vu over v's in-edges; w in CSR order, 64 bits."""
    n = a["n"]
    if "csc_off" in a:
        return _matrix(a["csc_off"], a["csc_idx"], w[a["perm"]], n)
    return _matrix(a["csr_off"], a["csr_idx"], w[_mirror(a)], n)


def _transition(a):
    """1 / out-degree per CSR edge."""
    deg = (a["csr_off"][1:] - a["csr_off"][:-1]).double()
    return torch.repeat_interleave(1.0 / deg.clamp(min=1), deg.long())


def _exact_rank(a, case):
    n, d = a["n"], float(np.float32(0.85))
    s = a["s"].double() if "s" in a else torch.full((n,), 1.0 / n, dtype=torch.float64, device=DEV)
    P = _in_edges(a, a["w"].double() if "w" in a else _transition(a))
    x = torch.full((n,), 1.0 / n, dtype=torch.float64, device=DEV)
    for _ in range(case["iters"]):
        y = (1 - d) * s + d * (P @ x)
        r = float((y - x).abs().sum()) if case["tol"] else 1.0
        x = y
        if r < case["tol"]:
            break
    return x


def _exact_grad(a, case):
    n, d = a["n"], float(np.float32(0.85))
    row = _rows(a)
    w = a["w"].double()
    total = torch.zeros(n, dtype=torch.float64, device=DEV).index_add_(0, row, w)
    inv = torch.where(total > 0, 1.0 / total.clamp(min=1e-300), torch.zeros_like(total))
    p = w * inv[row]
    P, PT = _in_edges(a, p), _matrix(a["csr_off"], a["csr_idx"], p, n)
    s, g = a["s"].double(), a["g"].double()
    x = torch.full((n,), 1.0 / n, dtype=torch.float64, device=DEV)
    lam = g.clone()
    for _ in range(case["iters"]):
        x = (1 - d) * s + d * (P @ x)
        lam = g + d * (PT @ lam)
    gw = (x * inv)[row] * (d * lam[a["csr_idx"].long()] - lam[row] + g[row])
    return {"ranks": x, "grad_w": gw, "grad_s": (1 - d) * lam}


def _exact_sssp(a):
    row, col, w = _rows(a), a["csr_idx"].long(), a["w"].double()
    dist = torch.full((a["n"],), math.inf, dtype=torch.float64, device=DEV)
    dist[int(a["sources"][0])] = 0.0
    while True:
        new = dist.clone().scatter_reduce_(0, col, dist[row] + w, "amin")
        if torch.equal(new, dist):
            return {"dist": dist, "pred": None}
        dist = new


def _exact_bc(a):
    n, row, col = a["n"], _rows(a), a["csr_idx"].long()
    total = torch.zeros(n, dtype=torch.float64, device=DEV)
    for src in a["sources"]:
        level = torch.full((n,), -1, dtype=torch.int32, device=DEV)
        sigma = torch.zeros(n, dtype=torch.float64, device=DEV)
        level[int(src)], sigma[int(src)] = 0, 1.0
        hops, depth = [], 0
        while True:
            e = torch.nonzero((level[row] == depth) & ((level[col] < 0) | (level[col] == depth + 1))).flatten()
            if not e.numel():
                break
            u, v = row[e], col[e]
            level[v] = depth + 1
            sigma.index_add_(0, v, sigma[u])
            hops.append((u, v))
            depth += 1
        delta = torch.zeros(n, dtype=torch.float64, device=DEV)
        for u, v in reversed(hops):
            delta.index_add_(0, u, sigma[u] / sigma[v] * (1.0 + delta[v]))
        delta[int(src)] = 0.0
        total += delta
    return total


def _exact_ppr(a, sources, tol):
    n, k, d = a["n"], len(sources), float(np.float32(0.85))
    P = _in_edges(a, _transition(a))
    e = torch.zeros((n, k), dtype=torch.float64, device=DEV)
    e[torch.as_tensor(sources, device=DEV).long(), torch.arange(k, device=DEV)] = 1.0
    x = e.clone()
    going = torch.arange(k, device=DEV)
    for _ in range(1000):
        xs = x[:, going]
        y = (1 - d) * e[:, going] + d * (P @ xs)
        r = (y - xs).abs().sum(0)
        x[:, going] = y
        going = going[r >= tol]
        if not going.numel():
            break
    return x


def exact(case, seed):
    what = case["what"]
    if what in ("bfs", "bfs_multi", "triangles", "msbfs"):  # whole numbers
        return None
    a = _inputs(case, seed)
    if what == "rank":
        return _exact_rank(a, case)
    if what == "grad":
        return _exact_grad(a, case)
    if what == "sssp":
        return _exact_sssp(a)
    if what == "bc":
        return _exact_bc(a)
    return [_exact_ppr(x, s, case["tol"]) for x, s in zip(a["graphs"], a["sources"])]
