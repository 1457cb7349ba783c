"""The one-block-per-source kernel (source.cu) against the CPU oracle, through
the C ABI, at the edges of its forms:

  * tau in 32-bit shared memory, in 16-bit shared memory (and sources whose
    distances pass 65534, redone in the wide form), in global memory;
  * arcs as packed words and without weights, the largest weights;
  * rows past the length that the block's warps share, and more of them in one
    step than its list holds;
  * buckets with more entries than their room, sources with more DAG arcs than
    are recorded;
  * a large graph with few sources, which keeps the distance step kernels.
Bars: tau and sigma_bar bit-exact, lambda within 1e-9 relative with exact zeros.
"""
import numpy as np
import pytest

import graphgen as gg
import oracle
import paper_1609_07008_gb300 as mfbc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1609_07008_gb300 import build
    build.build()
    mfbc.load()


def close(got, want, rtol=1e-9):
    got = np.asarray(got, np.float64)
    want = np.asarray(want, np.float64)
    zero = want == 0
    assert np.array_equal(got[zero], want[zero]), "exact zeros differ"
    rel = np.abs(got[~zero] - want[~zero]) / np.abs(want[~zero])
    assert rel.size == 0 or rel.max() <= rtol, f"max rel err {rel.max():.3e}"


def csr(n, u, v, w, directed):
    """CSRGraph of the arcs (u, v, w); undirected input holds each edge once."""
    if not directed:
        u, v, w = np.concatenate([u, v]), np.concatenate([v, u]), np.concatenate([w, w])
    key, at = np.unique(u.astype(np.int64) * n + v, return_index=True)
    rp = np.zeros(n + 1, np.int64)
    np.add.at(rp, key // n + 1, 1)
    return gg.CSRGraph(n=n, rowptr=np.cumsum(rp), col=(key % n).astype(np.int32), w=w[at].astype(np.int32),
                       directed=directed)


def with_tail(g, length, w):
    """g (undirected) with a path of `length` further vertices of weight w at vertex 0."""
    u = np.repeat(np.arange(g.n), g.out_degree())
    keep = u < g.col
    t = np.concatenate([[0], np.arange(g.n, g.n + length)])
    return csr(g.n + length, np.concatenate([u[keep], t[:-1]]), np.concatenate([g.col[keep], t[1:]]),
               np.concatenate([g.w[keep], np.full(length, w)]), False)


def torus(L, seed):
    """Directed arcs right, down and right-down on an L x L torus, weights U[1, 16]."""
    v = np.arange(L * L)
    r, c = v // L, v % L
    heads = [r * L + (c + 1) % L, (r + 1) % L * L + c, (r + 1) % L * L + (c + 1) % L]
    return csr(L * L, np.tile(v, 3), np.concatenate(heads), np.random.default_rng(seed).integers(1, 17, 3 * L * L), True)


def hubs(count, leaves, directed, seed):
    """Vertex 0 -> `count` hubs at one distance, every hub joined to every leaf."""
    rng = np.random.default_rng(seed)
    h = np.arange(1, count + 1)
    u = np.concatenate([np.zeros(count, np.int64), np.repeat(h, leaves)])
    v = np.concatenate([h, np.tile(np.arange(count + 1, count + 1 + leaves), count)])
    w = np.concatenate([np.full(count, 2), rng.integers(1, 4, count * leaves)])
    if directed:                                   # and some arcs back, so that other sources reach the hubs
        b = np.arange(count + 1, count + 1 + leaves, 7)
        u, v = np.concatenate([u, b]), np.concatenate([v, np.resize(h, len(b))])
        w = np.concatenate([w, rng.integers(1, 4, len(b))])
    return csr(count + 1 + leaves, u, v, w, directed)


def star(leaves, seed):
    n = leaves + 1
    rng = np.random.default_rng(seed)
    e = rng.integers(1, n, (2000, 2))
    e = e[e[:, 0] < e[:, 1]]
    u = np.concatenate([np.zeros(leaves, np.int64), e[:, 0]])
    v = np.concatenate([np.arange(1, n), e[:, 1]])
    return csr(n, u, v, np.concatenate([np.full(leaves, 3), rng.integers(1, 4, len(e))]), False)


CASES = {
    "smem32_directed": lambda: (gg.erdos_renyi(3001, 9, directed=True, weights=(1, 40), seed=3), 70),
    "smem32_one_block_an_sm": lambda: (gg.erdos_renyi(40001, 12, weights=(1, 20), seed=4), 9),
    "smem16": lambda: (gg.erdos_renyi(70001, 12, weights=(1, 30), seed=5), 20),
    "smem16_redone_wide": lambda: (with_tail(gg.erdos_renyi(60001, 12, weights=(1, 100), seed=6), 900, 100), 20),
    "global_lattice": lambda: (gg.grid2d(250, weights=(1, 16), seed=7), 170),
    "global_directed_lattice": lambda: (torus(250, 8), 160),
    "no_bucket_room_in_shared_memory": lambda: (gg.erdos_renyi(30001, 6, directed=True, weights=(1, 4096), seed=9), 20),
    "unit_weights": lambda: (gg.rmat(11, 8, seed=10), 50),
    "unit_weights_directed": lambda: (gg.rmat(11, 8, directed=True, seed=11), 50),
    "hub_list": lambda: (hubs(20, 700, False, 12), 40),
    "hub_list_overflows": lambda: (hubs(100, 600, False, 13), 30),
    "hub_list_overflows_directed": lambda: (hubs(100, 600, True, 14), 30),
    "bucket_overflows": lambda: (star(4000, 15), 40),
    "dag_overflows": lambda: (gg.erdos_renyi(300, 290, weights=(1, 2), seed=16), 40),
    "few_sources_wide_steps": lambda: (gg.erdos_renyi((1 << 18) + 3, 6, weights=(1, 9), seed=17), 5),
}


@pytest.mark.parametrize("name", CASES)
def test_forms_match_oracle(name):
    import torch
    g, k = CASES[name]()
    srcs = np.concatenate([[0], gg.sample_sources(g, k, seed=2)]).astype(np.int32)
    want = oracle.bc(g, srcs)
    wd, ws, _ = oracle.sssp(g, srcs[:20])
    G = mfbc.Graph.from_csr(g)
    try:
        paths = [mfbc.PATH_DIST] if g.w is None else [mfbc.PATH_AUTO, mfbc.PATH_DIST]
        for p in paths:
            close(G.bc(srcs, path=p), want)
            d, s = G.sssp(srcs[:20], path=p)
            assert np.array_equal(d, wd) and np.array_equal(s, ws)
        cut = len(srcs) // 3
        lists = [torch.from_numpy(x).cuda() for x in (srcs[:cut], srcs[cut:])]
        rows = G.bc_multi(lists, path=paths[-1], n_b=32).cpu().numpy()
        close(rows.sum(0), want)
        if cut:
            close(rows[0], oracle.bc(g, srcs[:cut]))
    finally:
        G.close()


def unit(g):
    return gg.CSRGraph(n=g.n, rowptr=g.rowptr, col=g.col, w=None, directed=g.directed)


# without weights: tau in 16-bit, 8-bit (a source deeper than 254 levels is redone
# wide) and global memory; more DAG arcs than are recorded; rows the warps share
UNIT_CASES = {
    "smem16": lambda: (gg.erdos_renyi(40001, 12, seed=21), 20),
    "smem16_directed": lambda: (gg.rmat(11, 8, directed=True, seed=22), 60),
    "smem8": lambda: (gg.erdos_renyi(120001, 10, seed=23), 9),
    "smem8_redone_wide": lambda: (unit(with_tail(gg.erdos_renyi(120001, 10, weights=(1, 2), seed=24), 300, 1)), 9),
    "global": lambda: (gg.erdos_renyi(120001, 4, seed=25), 9),
    "dag_overflows": lambda: (gg.erdos_renyi(300, 290, seed=26), 40),
    "hub_list_overflows": lambda: (unit(hubs(100, 600, False, 27)), 30),
    "hub_list_overflows_directed": lambda: (unit(hubs(100, 600, True, 28)), 30),
}


@pytest.mark.parametrize("name", UNIT_CASES)
def test_unit_forms_match_oracle(name):
    g, k = UNIT_CASES[name]()
    srcs = np.concatenate([[0], gg.sample_sources(g, k, seed=3)]).astype(np.int32)
    want = oracle.bc(g, srcs)
    wd, ws, _ = oracle.sssp(g, srcs[:20])
    G = mfbc.Graph.from_csr(g)
    try:
        for p in (mfbc.PATH_SMALL, mfbc.PATH_AUTO):
            close(G.bc(srcs, path=p), want)
            d, s = G.sssp(srcs[:20], path=p)
            assert np.array_equal(d, wd) and np.array_equal(s, ws)
    finally:
        G.close()


def test_workspaces_of_any_accepted_size():
    # a caller's workspace sized for many sources serves few, and one as small
    # as the narrowest width's serves all
    import torch
    g = gg.erdos_renyi(5000, 6, weights=(1, 9), seed=20)
    srcs = gg.sample_sources(g, 400, seed=1)
    want = oracle.bc(g, srcs)
    G = mfbc.Graph.from_csr(g)
    wide = torch.empty(G.workspace_size(400, 0), dtype=torch.uint8, device="cuda")
    close(G.bc(srcs, workspace=wide), want)
    close(G.bc(srcs[:3], workspace=wide), oracle.bc(g, srcs[:3]))
    narrow = torch.empty(G.workspace_size(400, 0, n_b=32), dtype=torch.uint8, device="cuda")
    close(G.bc(srcs, workspace=narrow, n_b=32), want)
    close(G.bc(srcs, workspace=narrow), want)
    G.close()


def test_threads_with_different_shared_memory_sizes():
    # one kernel form, two graphs whose blocks take different amounts of shared
    # memory, called from threads at the same time
    import threading
    import torch
    jobs = []
    for n, seed in ((300, 30), (3001, 31), (9001, 32), (16384, 33)):
        g = gg.erdos_renyi(n, 12, seed=seed)
        srcs = gg.sample_sources(g, 40, seed=1)
        jobs.append((mfbc.Graph.from_csr(g), torch.from_numpy(srcs).cuda(), oracle.bc(g, srcs)))
    failed = []

    def work(G, srcs, want):
        try:
            stream = torch.cuda.Stream()
            for _ in range(200):
                with torch.cuda.stream(stream):
                    lam = G.bc(srcs, stream=stream)
            stream.synchronize()
            close(lam.cpu().numpy(), want)
        except BaseException as e:
            failed.append(e)

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed[0]
    for G, _, _ in jobs:
        G.close()
