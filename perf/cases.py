"""The calls that a user of this framework makes, as measurable cases.

A case is one call (or, for "load", one graph and one call) through the public
entry points of paper_1609_07008_gb300 with the library's own choices of kernel
family and batch width:

  op "bc"     Graph.bc: betweenness summed over a list of sources;
  op "sssp"   Graph.sssp: distances and path counts, one row per source;
  op "multi"  Graph.bc_multi: several requests in one call, one row each;
  op "load"   Graph(...) from host CSR arrays, Graph.bc, close: what a program
              pays that gets a new graph and asks it once.

Graphs are the framework's own input families: R-MAT (quadrant probabilities
.57 / .19 / .19 / .05, relabelled at random, duplicates merged), uniform random
graphs of a given average degree, and 4-neighbour grids, with unit or integer
weights, undirected or directed.  They are generated on the GPU from the seed
and, but for "load", held as a Graph, which is what a program keeps.  "io" says
where the sources and the result live: "host" (numpy) or "device" (torch).
"""
import math

import numpy as np
import torch

import paper_1609_07008_gb300 as mfbc


def _case(name, op, graph, size, degree, sources, *, wmax=1, directed=False, io="device", requests=0):
    c = {"op": op, "graph": graph, "size": size, "degree": degree, "wmax": wmax, "directed": directed,
         "sources": sources, "requests": requests, "io": io}
    return dict(c, name=name) if name else c


def listed():
    return [
        # every vertex of a small network, arrays on the host: a script's first call
        _case("er1024_all_host", "bc", "er", 1024, 8, 1024, io="host"),
        # a few small requests on the smallest resident graph of a server: latency
        _case("rmat10_requests", "multi", "rmat", 10, 16, 400, requests=5),
        # a mid-size social-type graph, sampled sources, one ragged batch
        _case("rmat14", "bc", "rmat", 14, 16, 1000),
        # requests of mixed lengths packed into common batches on a resident graph
        _case("rmat16_requests", "multi", "rmat", 16, 16, 2500, requests=8),
        # a directed link graph
        _case("rmat17_directed", "bc", "rmat", 17, 16, 1500, directed=True),
        # the large power-law graph: the benchmark's shape at the largest size that is quick to set up
        _case("rmat20", "bc", "rmat", 20, 16, 4096),
        # a large uniform graph with an odd number of vertices
        _case("er300k", "bc", "er", 300007, 32, 2048),
        # distances and path counts alone (the forward direction), all rows returned
        _case("rmat18_sssp", "sssp", "rmat", 18, 16, 300),
        # a road-like weighted grid: many distance values, few arcs
        _case("grid256w", "bc", "grid", 256, 4, 512, wmax=16),
        # a dense weighted uniform graph
        _case("er32k_dense_w", "bc", "er", 32768, 512, 300, wmax=100),
        # a weighted directed power-law graph with hubs
        _case("rmat16w_directed", "bc", "rmat", 16, 16, 2048, wmax=255, directed=True),
        # a new graph from host arrays, asked once
        _case("rmat18_load", "load", "rmat", 18, 16, 256, io="host"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.randrange(9)
    io = rng.choice(["device", "host"])
    if kind == 0:      # small unit-weight graphs
        return _case(None, rng.choice(["bc", "sssp"]), "er", _log(rng, 200, 8000), rng.randint(3, 24),
                     _log(rng, 8, 180), io=io, directed=rng.random() < 0.3)
    if kind == 1:      # requests
        s = rng.randint(10, 17)
        return _case(None, "multi", "rmat", s, rng.randint(8, 18), _log(rng, 64, 3000 if s > 12 else 600),
                     requests=rng.randint(2, 9))
    if kind == 2:      # power-law graphs
        return _case(None, "bc", "rmat", rng.randint(13, 19), rng.randint(6, 20), _log(rng, 64, 4096), io=io)
    if kind == 3:      # directed power-law graphs
        return _case(None, "bc", "rmat", rng.randint(13, 18), rng.randint(6, 20), _log(rng, 64, 2500), io=io,
                     directed=True)
    if kind == 4:      # uniform graphs
        return _case(None, "bc", "er", _log(rng, 9000, 400000), rng.randint(6, 40), _log(rng, 64, 2500), io=io)
    if kind == 5:      # distances and path counts
        return _case(None, "sssp", "rmat", rng.randint(12, 18), rng.randint(6, 18), _log(rng, 16, 400),
                     directed=rng.random() < 0.3)
    if kind == 6:      # weighted grids
        return _case(None, rng.choice(["bc", "bc", "sssp"]), "grid", _log(rng, 40, 300), 4, _log(rng, 32, 600),
                     wmax=rng.randint(4, 16))
    if kind == 7:      # weighted uniform graphs, sparse to dense
        n = _log(rng, 2000, 40000)
        return _case(None, "bc", "er", n, _log(rng, 8, 512), _log(rng, 32, 300), wmax=rng.randint(10, 100), io=io)
    return _case(None, "bc", "rmat", rng.randint(11, 16), rng.randint(8, 18), _log(rng, 64, 2048),  # weighted hubs
                 wmax=rng.randint(32, 255), directed=rng.random() < 0.7, io=io)


# ----------------------------------------------------------------- inputs
_DEV = "cuda"


def _vertices(case):
    return {"rmat": 1 << case["size"], "er": case["size"], "grid": case["size"] ** 2}[case["graph"]]


def _edge_keys(case, n, gen):
    """Distinct (tail, head) pairs as tail * n + head; tail < head when undirected."""
    if case["graph"] == "grid":
        L = case["size"]
        v = torch.arange(n, device=_DEV)
        right, down = v[v % L < L - 1], v[v < n - L]
        return torch.cat([right * n + right + 1, down * n + down + L])
    if case["graph"] == "rmat":
        m = case["degree"] << case["size"]
        u = torch.zeros(m, dtype=torch.int64, device=_DEV)
        v = torch.zeros_like(u)
        for _ in range(case["size"]):
            r = torch.rand(m, device=_DEV, generator=gen)
            u = 2 * u + (r >= 0.76)
            v = 2 * v + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
        p = torch.randperm(n, device=_DEV, generator=gen)
        u, v = p[u], p[v]
    else:
        m = n * case["degree"] // (1 if case["directed"] else 2)
        u = torch.randint(n, (m,), device=_DEV, generator=gen)
        v = torch.randint(n, (m,), device=_DEV, generator=gen)
    ok = u != v
    u, v = u[ok], v[ok]
    if not case["directed"]:
        u, v = torch.minimum(u, v), torch.maximum(u, v)
    return torch.unique(u * n + v)


def _inputs(case, seed):
    """(n, rowptr int64, col int32, w int32 or None, sources int32, request offsets), on the GPU."""
    gen = torch.Generator(device=_DEV)
    gen.manual_seed(seed)
    n = _vertices(case)
    key = _edge_keys(case, n, gen)
    u, v = key // n, key % n
    w = None
    if case["wmax"] > 1:
        w = torch.randint(1, case["wmax"] + 1, (key.numel(),), device=_DEV, generator=gen, dtype=torch.int32)
    if not case["directed"]:
        u, v = torch.cat([u, v]), torch.cat([v, u])
        w = None if w is None else torch.cat([w, w])
    key, order = torch.sort(u * n + v)
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=_DEV)
    rowptr[1:] = torch.cumsum(torch.bincount(u, minlength=n), 0)
    col = (key % n).to(torch.int32)
    w = None if w is None else w[order].contiguous()
    cand = torch.nonzero(rowptr[1:] > rowptr[:-1]).reshape(-1)
    pick = torch.randperm(cand.numel(), device=_DEV, generator=gen)[: case["sources"]]
    src = cand[pick].to(torch.int32)
    off = np.array([0, src.numel()], dtype=np.int32)
    if case["requests"]:             # cut points spread over the logarithm: short and long requests
        share = np.exp(np.random.RandomState(seed % (1 << 31)).uniform(0.0, 3.0, case["requests"]))
        off = np.concatenate([[0], np.round(np.cumsum(share) / share.sum() * src.numel())]).astype(np.int32)
    return n, rowptr, col, w, src, off


def prepare(case, seed):
    n, rowptr, col, w, src, off = _inputs(case, seed)
    s = {"op": case["op"], "directed": case["directed"]}
    s["sources"] = src.cpu().numpy() if case["io"] == "host" else src
    if case["op"] == "multi":
        s["sources"] = [src[a:b].contiguous() for a, b in zip(off[:-1].tolist(), off[1:].tolist())]
    if case["op"] == "load":
        s["csr"] = (rowptr.cpu().numpy(), col.cpu().numpy(), None if w is None else w.cpu().numpy())
    else:
        s["graph"] = mfbc.Graph(rowptr, col, w, directed=case["directed"])
    return s


def run(state):
    if state["op"] == "load":
        with mfbc.Graph(*state["csr"], directed=state["directed"]) as g:
            return g.bc(state["sources"])
    if state["op"] == "sssp":
        return state["graph"].sssp(state["sources"])
    if state["op"] == "multi":
        return state["graph"].bc_multi(state["sources"])
    return state["graph"].bc(state["sources"])


def work(case):
    """The graph and the sources read once and the results written once; one
    operation per source and arc in each direction (the customary TEPS count)."""
    n = _vertices(case)
    if case["graph"] == "grid":
        nnz = 4 * n
    else:
        nnz = case["degree"] * n * (2 if case["graph"] == "rmat" and not case["directed"] else 1)
    k = min(case["sources"], n)
    out = 12.0 * n * k if case["op"] == "sssp" else 8.0 * n * max(1, case["requests"])
    return {"bytes": 4.0 * nnz * (2 if case["wmax"] > 1 else 1) + 8.0 * (n + 1) + 4.0 * k + out,
            "flops": float(nnz) * k * (1 if case["op"] == "sssp" else 2)}


# ------------------------------------------------ the same numbers in 64 bits
def _unit64(n, rowptr, col, src, on_block):
    """Breadth-first levels, path counts and dependencies of blocks of sources."""
    ones = torch.ones(col.numel(), dtype=torch.float64, device=_DEV)
    head = col.long()
    tail = torch.repeat_interleave(torch.arange(n, device=_DEV), rowptr[1:] - rowptr[:-1])
    A = torch.sparse_csr_tensor(rowptr, head, ones, (n, n))
    order = torch.argsort(head, stable=True)
    rpt = torch.zeros(n + 1, dtype=torch.int64, device=_DEV)
    rpt[1:] = torch.cumsum(torch.bincount(head, minlength=n), 0)
    At = torch.sparse_csr_tensor(rpt, tail[order], ones, (n, n))
    del head, tail, order
    B = 128 if n > 100000 else 256
    for b in range(0, src.numel(), B):
        s = src[b:b + B].long()
        j = torch.arange(s.numel(), device=_DEV)
        dist = torch.full((n, s.numel()), -1, dtype=torch.int32, device=_DEV)
        sig = torch.zeros(n, s.numel(), dtype=torch.float64, device=_DEV)
        dist[s, j], sig[s, j] = 0, 1.0
        front, depth = sig.clone(), 0
        while True:
            front = (At @ front).masked_fill_(dist >= 0, 0.0)
            new = front > 0
            if not bool(new.any()):
                break
            depth += 1
            dist.masked_fill_(new, depth)
            sig += front
        zeta = torch.zeros_like(sig)
        inv = torch.where(sig > 0, 1.0 / sig, sig)
        if on_block.needs_zeta:
            for d in range(depth, 1, -1):
                val = torch.where(dist == d, zeta + inv, 0.0)
                zeta += (A @ val).masked_fill_(dist != d - 1, 0.0)
        on_block(b, s, dist, sig, zeta)


def _weighted64(n, rowptr, col, w, src, on_block):
    """The same for integer weights: distances to their fixed point, then counts
    and dependencies over the tight arcs, as many rounds as the longest path has arcs."""
    deg = rowptr[1:] - rowptr[:-1]
    head, wt = col.long(), w.to(torch.float64)
    tail = torch.repeat_interleave(torch.arange(n, device=_DEV), deg)
    D = int(deg.max())
    grid = D <= 8                    # few arcs a row (undirected): one gather for each arc place
    if grid:
        at = rowptr[:-1, None] + torch.arange(D, device=_DEV)[None, :]
        has = torch.arange(D, device=_DEV)[None, :] < deg[:, None]
        at = torch.where(has, at, 0)
        nbr = head[at]
        nw = torch.where(has, wt[at], math.inf)
    B = max(8, min(512, (1 << 29) // max(1, n if grid else head.numel())))
    for b in range(0, src.numel(), B):
        s = src[b:b + B].long()
        k = s.numel()
        j = torch.arange(k, device=_DEV)
        dist = torch.full((n, k), math.inf, dtype=torch.float64, device=_DEV)
        dist[s, j] = 0.0
        while True:
            if grid:
                new = dist.clone()
                for d in range(D):
                    new = torch.minimum(new, dist[nbr[:, d]] + nw[:, d, None])
            else:
                new = dist.scatter_reduce(0, head[:, None].expand(-1, k), dist[tail] + wt[:, None], "amin")
            if torch.equal(new, dist):
                break
            dist = new
        reach = torch.isfinite(dist)
        seed = torch.zeros_like(dist)
        seed[s, j] = 1.0

        def pull(x, backward):       # sum of x over the tight arcs that end (backward: start) at a vertex
            y = torch.zeros_like(x)
            if grid:
                for d in range(D):
                    o = nbr[:, d]
                    step = dist[o] - dist if backward else dist - dist[o]
                    y += torch.where(step == nw[:, d, None], x[o], 0.0)
                return y
            tight = dist[tail] + wt[:, None] == dist[head]
            tight &= reach[tail]
            one, other = (tail, head) if backward else (head, tail)
            return y.index_add_(0, one, torch.where(tight, x[other], 0.0))

        sig, rounds = seed, 0
        while True:
            new = torch.where(reach, pull(sig, False), 0.0) + seed
            if torch.equal(new, sig):
                break
            sig, rounds = new, rounds + 1
        zeta = torch.zeros_like(sig)
        inv = torch.where(sig > 0, 1.0 / sig, 0.0)
        if on_block.needs_zeta:
            for _ in range(rounds):
                zeta = torch.where(reach, pull(zeta + inv, True), 0.0)
        on_block(b, s, torch.where(reach, dist, 2147483647.0).to(torch.int32), sig, zeta)


class _Rows:
    needs_zeta = False

    def __init__(self, n, k):
        self.dist = torch.empty((k, n), dtype=torch.int32, device=_DEV)
        self.sig = torch.empty((k, n), dtype=torch.float64, device=_DEV)

    def __call__(self, b, s, dist, sig, zeta):
        self.dist[b:b + s.numel()] = torch.where(dist < 0, 2147483647, dist).t()
        self.sig[b:b + s.numel()] = sig.t()


class _Lambda:
    needs_zeta = True

    def __init__(self, n, off):
        self.lam = torch.zeros((len(off) - 1, n), dtype=torch.float64, device=_DEV)
        self.off = off

    def __call__(self, b, s, dist, sig, zeta):
        term = zeta * sig
        term[s, torch.arange(s.numel(), device=_DEV)] = 0.0
        for r in range(len(self.off) - 1):
            lo, hi = max(int(self.off[r]) - b, 0), min(int(self.off[r + 1]) - b, s.numel())
            if lo < hi:
                self.lam[r] += term[:, lo:hi].sum(1)


def exact(case, seed):
    n, rowptr, col, w, src, off = _inputs(case, seed)
    rows = _Rows(n, src.numel()) if case["op"] == "sssp" else _Lambda(n, off)
    if w is None:
        _unit64(n, rowptr, col, src, rows)
    else:
        _weighted64(n, rowptr, col, w, src, rows)
    if case["op"] == "sssp":
        return (rows.dist, rows.sig) if case["io"] == "device" else (rows.dist.cpu().numpy(), rows.sig.cpu().numpy())
    lam = rows.lam if case["op"] == "multi" else rows.lam[0]
    return lam.cpu().numpy() if case["io"] == "host" else lam
