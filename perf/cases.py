"""Performance cases: the work that a user of the library has it do, through
its public entry points (paper_0809_1906_gb300.native and the C ABI behind it).

Graphs are seeded and synthetic, built on the GPU with torch, and handed over
as host CSR arrays. The families and sizes follow the repository's own
workloads (graphs.py, bench.py): R-MAT, sparse random graphs, meshes with
long-range edges (weighted and not), dense G(n, p) and sets of many small
graphs. An unweighted or weighted pass is one bc_run and the read of its
result (and of the per-source summaries where a case asks for them).
"""
import math

import numpy as np
import torch

from paper_0809_1906_gb300 import native

DEV = "cuda"

# Mean undirected degree of an R-MAT graph without its isolated vertices (edge
# factor 16, duplicates dropped): about 2 m / n at the sizes used here.
_RMAT_DEGREE = 38.0


def listed():
    return [
        # One small graph, every vertex a source, halved for unordered pairs:
        # the smallest everyday call, bound by launches and host steps.
        {"name": "small_random_300", "kind": "random", "n": 300, "m": 1000, "sources": 0, "halve": True,
         "summaries": False},
        # G(n, 4n) plus a Hamiltonian path, every vertex a source, summaries read.
        {"name": "random_1024", "kind": "random", "n": 1024, "m": 4096, "sources": 0, "halve": False,
         "summaries": True},
        # The headline workload: a skewed (social or web like) graph, exact
        # betweenness from every vertex.
        {"name": "rmat_s16_all", "kind": "rmat", "scale": 16, "directed": False, "sources": 0, "summaries": False},
        # A directed skewed graph (citations, links), every vertex a source.
        {"name": "rmat_s14_directed_all", "kind": "rmat", "scale": 14, "directed": True, "sources": 0,
         "summaries": False},
        # A larger skewed graph with sampled sources, as approximate
        # betweenness uses; the last batch is ragged.
        {"name": "rmat_s18_sampled_1000", "kind": "rmat", "scale": 18, "directed": False, "sources": 1000,
         "summaries": True},
        # An unweighted mesh with some long-range edges (road or power grid
        # like): many narrow levels, low degree.
        {"name": "mesh_128_all", "kind": "mesh", "side": 128, "frac": 0.05, "wmax": 0, "directed": False,
         "sources": 0, "summaries": False},
        # A weighted mesh (road lengths), sampled sources of a large graph.
        {"name": "weighted_mesh_512_sampled_4096", "kind": "mesh", "side": 512, "frac": 0.05, "wmax": 100,
         "directed": False, "sources": 4096, "summaries": False},
        # A small weighted mesh, every vertex a source.
        {"name": "weighted_mesh_64_all", "kind": "mesh", "side": 64, "frac": 0.05, "wmax": 100, "directed": False,
         "sources": 0, "summaries": True},
        # A dense graph, every vertex a source, on the tensor-core form.
        {"name": "dense_8192_all", "kind": "dense", "n": 8192, "p": 0.05, "wmax": 0},
        # A dense weighted graph of an odd size: distance products and the
        # pair formula.
        {"name": "dense_weighted_2001_all", "kind": "dense", "n": 2001, "p": 0.05, "wmax": 10},
        # A set of many small graphs of mixed sizes (ego networks, molecules,
        # circuit blocks): one plan, replayed.
        {"name": "many_1000", "kind": "many", "count": 1000, "nmin": 50, "nmax": 5000, "batch": 256},
        # The forward direction alone: distance and path-count rows of sampled
        # sources, left on the device.
        {"name": "rows_rmat_s15_512", "kind": "rows", "scale": 15, "sources": 512},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above."""
    kind = rng.choice(["random", "rmat", "rmat", "mesh", "weighted_mesh", "weighted_mesh", "dense", "dense_weighted",
                       "many", "rows"])
    if kind == "random":
        n = _log(rng, 200, 6000)
        return {"kind": "random", "n": n, "m": n * rng.randint(2, 6) + rng.randint(0, 99),
                "sources": rng.choice([0, 0, _log(rng, 33, n - 1)]), "halve": rng.random() < 0.5,
                "summaries": rng.random() < 0.5}
    if kind == "rmat":
        scale = rng.randint(12, 18)
        most = 30000 if scale < 16 else 4000 if scale < 18 else 1000
        every = scale < 15 and rng.random() < 0.5
        sources = 0 if every else min(_log(rng, 100, most), (1 << scale) // 4)
        return {"kind": "rmat", "scale": scale, "directed": rng.random() < 0.4,
                "sources": sources, "summaries": rng.random() < 0.5}
    if kind in ("mesh", "weighted_mesh"):
        side = _log(rng, 20, 160 if kind == "mesh" else 400)
        every = side <= 72 or (kind == "mesh" and side <= 128)
        return {"kind": "mesh", "side": side, "frac": round(rng.uniform(0.03, 0.2), 3),
                "wmax": 0 if kind == "mesh" else _log(rng, 2, 200), "directed": rng.random() < 0.25,
                "sources": 0 if every and rng.random() < 0.5 else min(_log(rng, 40, 3000), side * side),
                "summaries": rng.random() < 0.5}
    if kind == "dense":
        return {"kind": "dense", "n": _log(rng, 600, 8192), "p": round(rng.uniform(0.02, 0.12), 3), "wmax": 0}
    if kind == "dense_weighted":
        return {"kind": "dense", "n": _log(rng, 200, 2600), "p": round(rng.uniform(0.04, 0.12), 3),
                "wmax": rng.randint(2, 40)}
    if kind == "many":
        nmin = _log(rng, 20, 200)
        return {"kind": "many", "count": _log(rng, 50, 900), "nmin": nmin, "nmax": nmin * rng.randint(4, 20),
                "batch": rng.choice([64, 128, 256])}
    scale = rng.randint(11, 16)
    return {"kind": "rows", "scale": scale, "sources": _log(rng, 40, min(700, 1 << (scale - 2)))}


# ------------------------------------------------------------------- graphs

def _gen(seed, tag):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + tag) & 0x7FFFFFFFFFFFFFFF)
    return g


def _below(k, bound, g):
    return torch.randint(0, bound, (k,), generator=g, device=DEV)


def _csr(n, u, v, w=None, directed=False):
    """CSR (device int64: row_ptr, src, col, w) from distinct arcs or edges."""
    if not directed:
        u, v = torch.cat([u, v]), torch.cat([v, u])
        w = None if w is None else torch.cat([w, w])
    order = torch.argsort(u * n + v)
    u, v = u[order], v[order]
    rp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rp[1:] = torch.cumsum(torch.bincount(u, minlength=n), 0)
    return n, rp, u, v, None if w is None else w[order]


def _unique_edges(n, u, v):
    """Distinct undirected edges without loops, u < v."""
    keep = u != v
    key = torch.unique(torch.minimum(u, v)[keep] * n + torch.maximum(u, v)[keep])
    return key // n, key % n


def _random_edges(n, m, g):
    """About m uniform random edges plus a random Hamiltonian path."""
    u, v = _below(m, n, g), _below(m, n, g)
    perm = torch.randperm(n, generator=g, device=DEV)
    return _unique_edges(n, torch.cat([u, perm[:-1]]), torch.cat([v, perm[1:]]))


def _attachment_edges(n, g):
    """Preferential attachment, three arcs per new vertex: arc 3 i + j of vertex
    i picks a uniform earlier endpoint slot; picks that name another arc's
    target are followed to it."""
    arcs = 3 * (n - 1)
    src = torch.arange(1, n, device=DEV).repeat_interleave(3)
    r = torch.rand(arcs, generator=g, device=DEV, dtype=torch.float64)
    first = 6 * (src - 1)  # endpoint slots of the vertices before this one
    slot = torch.minimum((r * torch.clamp(first, min=1)).long(), torch.clamp(first - 1, min=0))
    tgt = torch.where(first == 0, 0, torch.where(slot % 2 == 0, src[slot // 2], -1))
    ref = slot // 2
    while bool((tgt < 0).any()):
        tgt = torch.where(tgt < 0, tgt[ref], tgt)
        ref = ref[ref]
    return _unique_edges(n, src, tgt)


def _core_size(scale):
    """Vertices kept of an R-MAT draw: about those of its largest component."""
    return int((0.95 - 0.015 * scale) * (1 << scale))


def _core(n, u, v, size):
    """New id of each of the `size` vertices with the most arcs (ties by id), else -1."""
    deg = torch.bincount(torch.cat([u, v]), minlength=n)
    best = torch.sort(deg, descending=True, stable=True).indices[:size]
    inside = torch.zeros(n, dtype=torch.bool, device=DEV)
    inside[best] = True
    return torch.where(inside, torch.cumsum(inside.long(), 0) - 1, -1)


def _rmat(scale, directed, seed):
    """R-MAT (0.57, 0.19, 0.19, 0.05), edge factor 16, without its isolated fringe."""
    n, ne, g = 1 << scale, 16 << scale, _gen(seed, 1)
    u = torch.zeros(ne, dtype=torch.int64, device=DEV)
    v = torch.zeros(ne, dtype=torch.int64, device=DEV)
    for bit in range(scale):
        r = torch.rand(ne, generator=g, device=DEV, dtype=torch.float64)
        u |= (r >= 0.76).long() << bit
        v |= (((r >= 0.57) & (r < 0.76)) | (r >= 0.95)).long() << bit
    perm = torch.randperm(n, generator=g, device=DEV)
    u, v = perm[u], perm[v]
    if directed:
        key = torch.unique((u * n + v)[u != v])
        u, v = key // n, key % n
    else:
        u, v = _unique_edges(n, u, v)
    size = _core_size(scale)
    ids = _core(n, u, v, size)
    keep = (ids[u] >= 0) & (ids[v] >= 0)
    return _csr(size, ids[u[keep]], ids[v[keep]], directed=directed)


def _mesh(side, frac, wmax, directed, seed):
    """side x side grid plus frac of its edges at random, weights 1..wmax (0:
    none). Directed: every edge becomes two arcs, weighted apart, and one in
    eight arcs is closed."""
    n, g = side * side, _gen(seed, 2)
    at = torch.arange(n, device=DEV)
    right, down = at[at % side < side - 1], at[at < n - side]
    k = int(round(frac * 2 * side * (side - 1)))
    u = torch.cat([right, down, _below(k, n, g)])
    v = torch.cat([right + 1, down + side, _below(k, n, g)])
    u, v = _unique_edges(n, u, v)
    if directed:
        u, v = torch.cat([u, v]), torch.cat([v, u])
        keep = torch.rand(u.numel(), generator=g, device=DEV) >= 0.125
        u, v = u[keep], v[keep]
    w = _below(u.numel(), wmax, g) + 1 if wmax else None
    return _csr(n, u, v, w, directed)


def _dense(n, p, wmax, seed):
    """G(n, p), weights 1..wmax (0: none)."""
    g = _gen(seed, 3)
    hit = torch.rand((n, n), generator=g, device=DEV) < p
    u, v = torch.nonzero(torch.triu(hit, 1), as_tuple=True)
    return _csr(n, u, v, _below(u.numel(), wmax, g) + 1 if wmax else None)


def _many(case, seed):
    """Sizes log-uniform in [nmin, nmax]; random and preferential-attachment graphs in turn."""
    lo, hi = math.log(case["nmin"]), math.log(case["nmax"])
    sizes = np.rint(np.exp(np.random.default_rng(case["count"]).uniform(lo, hi, case["count"]))).astype(np.int64)
    g = _gen(seed, 4)
    for i, n in enumerate(sizes.tolist()):
        yield _csr(n, *(_random_edges(n, 3 * n, g) if i % 2 == 0 else _attachment_edges(n, g)))


def _graph(case, seed):
    if case["kind"] == "random":
        return _csr(case["n"], *_random_edges(case["n"], case["m"], _gen(seed, 5)))
    if case["kind"] in ("rmat", "rows"):
        return _rmat(case["scale"], case.get("directed", False), seed)
    if case["kind"] == "mesh":
        return _mesh(case["side"], case["frac"], case["wmax"], case["directed"], seed)
    return _dense(case["n"], case["p"], case["wmax"], seed)


def _sources(case, n, seed):
    """Distinct sampled source ids (host int32), or None for every vertex."""
    k = min(case.get("sources", 0), n)
    return np.random.default_rng(int(seed) + 7).permutation(n)[:k].astype(np.int32) if k else None


def _handle(csr, directed=False, trusted=False):
    n, rp, _, col, w = csr
    host = [None if x is None else x.to(torch.int32).cpu().numpy() for x in (rp, col, w)]
    return native.Graph(n, *host, directed=directed, trust_input=trusted)


# -------------------------------------------------------------------- cases

def prepare(case, seed):
    if case["kind"] == "many":
        graphs = [_handle(c, trusted=True) for c in _many(case, seed)]
        at = np.concatenate([[0], np.cumsum([g.n for g in graphs])])
        return {"kind": "many", "graphs": graphs, "plan": native.ManyPlan(graphs, batch=case["batch"]),
                "at": at.tolist(), "bc": np.empty(int(at[-1]), np.float64)}
    csr = _graph(case, seed)
    n = csr[0]
    state = {"kind": case["kind"], "graph": _handle(csr, case.get("directed", False)), "n": n,
             "sources": _sources(case, n, seed), "summaries": case.get("summaries", False), "flags": 0}
    if case["kind"] == "rows":
        k = len(state["sources"])
        state["sigma"] = torch.empty((k, n), dtype=torch.int64, device=DEV)
        state["dist"] = torch.empty((k, n), dtype=torch.int32, device=DEV)
        return state
    if case["kind"] == "dense":
        state["flags"] |= native.BC_DENSE
    if case.get("halve"):
        state["flags"] |= native.BC_HALVE
    state["bc"] = torch.empty(n, dtype=torch.float64, device=DEV)
    return state


def run(state):
    if state["kind"] == "many":
        state["plan"].run()
        state["plan"].result()
        at, bc = state["at"], state["bc"]
        for i, g in enumerate(state["graphs"]):
            g.result(out=bc[at[i]:at[i + 1]])
        return {"bc": bc}
    g = state["graph"]
    if state["kind"] == "rows":
        src = state["sources"]
        code = g.lib.bc_forward_rows(g.handle, src.ctypes.data, len(src), state["sigma"].data_ptr(),
                                     state["dist"].data_ptr(), None, torch.cuda.current_stream().cuda_stream)
        if code < 0:
            raise native.BcError(code, "bc_forward_rows", g.lib.bc_last_error().decode())
        return {"sigma": state["sigma"], "dist": state["dist"]}
    g.run(state["sources"], flags=state["flags"])
    g.result(out=state["bc"])
    out = {"bc": state["bc"]}
    if state["summaries"]:
        k = state["n"] if state["sources"] is None else len(state["sources"])
        out.update((name, x.view(np.int64)) for name, x in g.source_hashes(k).items())
    return out


def work(case):
    """Each pass visits every arc of every source once forward and once back
    (an add each); the CSR is read once and the result written once."""
    kind = case["kind"]
    if kind == "many":
        lo, hi = math.log(case["nmin"]), math.log(case["nmax"])
        mean = (case["nmax"] - case["nmin"]) / (hi - lo)
        square = (case["nmax"] ** 2 - case["nmin"] ** 2) / (2 * (hi - lo))
        return {"bytes": case["count"] * mean * (4 + 4 * 7 + 8), "flops": case["count"] * square * 7 * 2}
    weight = 1
    if kind == "random":
        n, arcs = case["n"], 2 * (case["m"] + case["n"])
    elif kind in ("rmat", "rows"):
        n = _core_size(case["scale"])
        arcs = n * _RMAT_DEGREE * (0.55 if case.get("directed") else 1.0)
    elif kind == "mesh":
        n = case["side"] ** 2
        arcs = 4 * n * (1 + case["frac"]) * (0.875 if case["directed"] else 1.0)
        weight = 2 if case["wmax"] else 1
    else:
        n = case["n"]
        arcs = n * n * case["p"]
        weight = 2 if case["wmax"] else 1
    nsrc = min(case.get("sources", 0), n) or n
    graph = 4 * (n + 1) + 4 * arcs * weight
    if kind == "rows":
        return {"bytes": graph + 12.0 * nsrc * n, "flops": float(nsrc) * arcs}
    return {"bytes": graph + 8.0 * n + (32.0 * nsrc if case.get("summaries") else 0.0),
            "flops": 2.0 * nsrc * arcs}


# ------------------------------------------------- the same answer in 64 bits

def _exact_levels(csr, sources):
    """Brandes level by level, a block of sources at a time, in FP64."""
    n, rp, src, col, _ = csr
    out = torch.sparse_csr_tensor(rp, col, torch.ones(col.numel(), dtype=torch.float64, device=DEV), (n, n))
    order = torch.argsort(col * n + src)
    rin = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rin[1:] = torch.cumsum(torch.bincount(col, minlength=n), 0)
    into = torch.sparse_csr_tensor(rin, src[order], torch.ones(col.numel(), dtype=torch.float64, device=DEV), (n, n))
    bc = torch.zeros(n, dtype=torch.float64, device=DEV)
    block = max(64, min(2048, (1 << 24) // max(n, 1)))
    for b0 in range(0, sources.numel(), block):
        s = sources[b0:b0 + block]
        cols = torch.arange(s.numel(), device=DEV)
        sigma = torch.zeros((n, s.numel()), dtype=torch.float64, device=DEV)
        level = torch.full((n, s.numel()), -1, dtype=torch.int32, device=DEV)
        sigma[s, cols] = 1.0
        level[s, cols] = 0
        depth, front = 0, sigma.clone()
        while True:
            nxt = torch.where(level < 0, into @ front, 0.0)
            hit = nxt > 0
            if not bool(hit.any()):
                break
            depth += 1
            level[hit] = depth
            sigma += nxt
            front = nxt
        c = torch.zeros_like(sigma)
        for lv in range(depth, 0, -1):
            here = level == lv
            total = torch.where(here, out @ c, 0.0)
            bc += (sigma * total).sum(1)
            c = torch.where(here, total + 1.0 / sigma, 0.0)
    return bc


def _exact_weighted(csr, sources):
    """Distances by relaxing every arc until nothing changes, then counts and
    dependencies over the arcs that lie on shortest paths, in FP64."""
    n, _, src, dst, w = csr
    bc = torch.zeros(n, dtype=torch.float64, device=DEV)
    block = max(16, min(1024, (1 << 26) // max(1, src.numel())))
    far = 1 << 30
    w = w.to(torch.int32)[:, None]
    for b0 in range(0, sources.numel(), block):
        s = sources[b0:b0 + block]
        cols = torch.arange(s.numel(), device=DEV)
        dist = torch.full((n, s.numel()), far, dtype=torch.int32, device=DEV)
        dist[s, cols] = 0
        heads = dst[:, None].expand(-1, s.numel())
        while True:
            new = dist.scatter_reduce(0, heads, dist[src] + w, "amin")
            new = torch.minimum(new, torch.tensor(far, dtype=torch.int32, device=DEV))
            if torch.equal(new, dist):
                break
            dist = new
        on = ((dist[src] + w) == dist[dst]).to(torch.float64)
        start = torch.zeros((n, s.numel()), dtype=torch.float64, device=DEV)
        start[s, cols] = 1.0
        sigma, steps = start, 0
        while True:
            new = start.index_add(0, dst, sigma[src] * on)
            steps += 1
            if bool(((new - sigma).abs() <= 1e-14 * new).all()):
                break
            sigma = new
        own = torch.where(sigma > 0, 1.0 / sigma, 0.0)
        total = torch.zeros_like(own)
        for _ in range(steps):
            total = torch.zeros_like(own).index_add(0, src, (own + total)[dst] * on)
        delta = sigma * total
        delta[s, cols] = 0.0
        bc += delta.sum(1)
    return bc


def _exact_bc(csr, sources):
    src = torch.arange(csr[0], device=DEV) if sources is None else torch.from_numpy(sources).to(DEV).long()
    return _exact_levels(csr, src) if csr[4] is None else _exact_weighted(csr, src)


def exact(case, seed):
    """Betweenness in FP64 with torch alone; None where that takes too long,
    and for the whole-number outputs."""
    kind = case["kind"]
    if kind == "rows":
        return None
    if kind == "many":
        return {"bc": torch.cat([_exact_bc(c, None) for c in _many(case, seed)])}
    if kind == "mesh" and case["wmax"]:
        nsrc = min(case["sources"] or case["side"] ** 2, case["side"] ** 2)
        if 4.2 * case["side"] ** 2 * nsrc * case["side"] > 6e10:
            return None
    csr = _graph(case, seed)
    bc = _exact_bc(csr, _sources(case, csr[0], seed))
    out = {"bc": bc / 2 if case.get("halve") else bc}
    if case.get("summaries"):
        out.update(hash_sigma=None, hash_dist=None, dist_sum=None, reach=None)
    return out
