"""Which kernels take a call: one block per source, or the family's own kernels
over the whole device.  Both give the same results; the choice decides the time,
so these cases lie where one side is well over 1.5 times faster.

Seen in the call's profile: "dist_mfbr" and "small_persistent" with one step a
batch are the families' kernels (the source kernel runs MFBr inside its one
launch).  Bars: tau and sigma_bar bit-exact, lambda within 1e-9 relative with
exact zeros, against the CPU oracle.
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


def permutations(n, count, wmax, seed):
    """Directed union of random permutations: in- and out-degrees at most `count`."""
    rng = np.random.default_rng(seed)
    key = np.unique(np.concatenate([np.arange(n) * n + rng.permutation(n) for _ in range(count)]))
    key = key[key // n != key % n]
    rowptr = np.zeros(n + 1, np.int64)
    rowptr[1:] = np.cumsum(np.bincount(key // n, minlength=n))
    return gg.CSRGraph(n=n, rowptr=rowptr, col=(key % n).astype(np.int32),
                       w=rng.integers(1, wmax + 1, len(key)).astype(np.int32), directed=True)


# graph, sources, by the step kernels of the distance family?
DIST_ROUTES = {
    "low_degrees_few_wide_steps": (lambda: permutations(1 << 18, 3, 16, 1), 1, True),
    "low_degrees_many_sources": (lambda: permutations(1 << 18, 3, 16, 1), 64, False),
    "lattice_one_source": (lambda: gg.grid2d(512, weights=(1, 16), seed=2), 1, False),
    "dense_few_sources": (lambda: gg.erdos_renyi(1 << 17, 64, weights=(1, 4), seed=3), 8, True),
    "sparse_many_distances": (lambda: gg.erdos_renyi(1 << 16, 6, weights=(1, 100), seed=4), 2, False),
    "below_the_line": (lambda: gg.erdos_renyi(20000, 12, weights=(1, 4), seed=5), 1, False),
}


@pytest.mark.parametrize("name", DIST_ROUTES)
def test_few_sources_of_weighted_graphs(name):
    make, k, steps = DIST_ROUTES[name]
    g = make()
    srcs = gg.sample_sources(g, k, seed=6)
    G = mfbc.Graph.from_csr(g)
    try:
        lam, prof = G.bc(srcs, profile=True)
        assert prof["path"] == mfbc.PATH_DIST
        assert ("dist_mfbr" in prof["kernels"]) == steps
        close(lam, oracle.bc(g, srcs))
        d, s = G.sssp(srcs[:2])
        wd, ws, _ = oracle.sssp(g, srcs[:2])
        assert np.array_equal(d, wd) and np.array_equal(s, ws)
    finally:
        G.close()


# unit weights past the small family: graph, sources, by the level kernels?
LEVEL_ROUTES = {
    "dense_one_source": (lambda: gg.erdos_renyi(9000, 65, seed=12), 1, True),
    "dense_fewer_arcs": (lambda: gg.erdos_renyi(9000, 33, seed=13), 1, False),
    "directed_one_source": (lambda: gg.erdos_renyi(16384, 35, directed=True, seed=14), 1, True),
    "sparse_one_source": (lambda: gg.erdos_renyi(400000, 3, seed=15), 1, True),
    "sparse_more_sources": (lambda: gg.erdos_renyi(400000, 3, seed=15), 40, False),
    "deep_one_source": (lambda: gg.grid2d(256, seed=16), 1, False),
}


@pytest.mark.parametrize("name", LEVEL_ROUTES)
def test_few_sources_of_unit_weight_graphs(name):
    make, k, levels = LEVEL_ROUTES[name]
    g = make()
    g = gg.CSRGraph(n=g.n, rowptr=g.rowptr, col=g.col, w=None, directed=g.directed)
    srcs = gg.sample_sources(g, k, seed=17)
    G = mfbc.Graph.from_csr(g)
    try:
        lam, prof = G.bc(srcs, profile=True)
        assert prof["path"] == mfbc.PATH_LEVEL
        assert ("level_mfbf_gather" in prof["kernels"]) == levels
        close(lam, oracle.bc(g, srcs))
    finally:
        G.close()


# graph, sources, n_b, path, by source?  (n_b = 32 leaves the source kernel a few
# blocks, 64 a block a column)
def _unit_rmat():
    return gg.rmat(12, 8, seed=7)


NARROW_ROUTES = {
    "dist_uniform_32": (lambda: gg.erdos_renyi(50000, 16, weights=(1, 20), seed=8), 48, 32, mfbc.PATH_AUTO, False),
    "dist_uniform_64": (lambda: gg.erdos_renyi(50000, 16, weights=(1, 20), seed=8), 64, 64, mfbc.PATH_AUTO, True),
    "dist_lattice_32": (lambda: gg.grid2d(200, weights=(1, 16), seed=9), 48, 32, mfbc.PATH_AUTO, True),
    "general_uniform_32": (lambda: gg.erdos_renyi(50000, 8, weights=(1, 255), seed=10), 300, 32, mfbc.PATH_AUTO, False),
    "general_hubs_64": (lambda: gg.rmat(15, 16, directed=True, weights=(1, 255), seed=10), 300, 64, mfbc.PATH_AUTO, True),
    "small_32_many": (_unit_rmat, 1000, 32, mfbc.PATH_SMALL, False),
    "small_32_few": (_unit_rmat, 8, 32, mfbc.PATH_SMALL, True),
    "small_64": (_unit_rmat, 1000, 64, mfbc.PATH_SMALL, True),
}


def by_source(prof):
    if prof["path"] == mfbc.PATH_SMALL:          # (the persistent kernel counts one step a batch)
        return prof["fwd_iters"] != prof["batches"]
    return not any(k in prof["kernels"] for k in ("dist_mfbr", "mfbf_accumulate", "level_mfbf_gather"))


@pytest.mark.parametrize("name", NARROW_ROUTES)
def test_narrow_batches_and_short_workspaces(name):
    import torch
    make, k, n_b, path, want_source = NARROW_ROUTES[name]
    g = make()
    srcs = gg.sample_sources(g, k, seed=11)
    want = oracle.bc(g, srcs)
    wd, ws, _ = oracle.sssp(g, srcs[:40])
    G = mfbc.Graph.from_csr(g)
    try:
        lam, prof = G.bc(srcs, n_b=n_b, path=path, profile=True)
        assert by_source(prof) == want_source
        close(lam, want)
        # the same calls in a workspace of the size asked for, and n_b = 0 in it
        work = torch.empty(G.workspace_size(k, 0, n_b=n_b, path=path), dtype=torch.uint8, device="cuda")
        lam, prof = G.bc(srcs, n_b=n_b, path=path, workspace=work, profile=True)
        assert by_source(prof) == want_source
        close(lam, want)
        close(G.bc(srcs, path=path, workspace=work), want)
        for rows in (1, 40):
            work = torch.empty(G.workspace_size(rows, 1, n_b=n_b, path=path), dtype=torch.uint8, device="cuda")
            d, s = G.sssp(srcs[:rows], n_b=n_b, path=path, workspace=work)
            assert np.array_equal(d, wd[:rows]) and np.array_equal(s, ws[:rows])
        cut = k // 3
        lists = [torch.from_numpy(x).cuda() for x in (srcs[:cut], srcs[cut:])]
        cols = sum((len(x) + 31) // 32 * 32 for x in lists)
        work = torch.empty(G.workspace_size(cols, 2, n_b=n_b, path=path), dtype=torch.uint8, device="cuda")
        close(G.bc_multi(lists, n_b=n_b, path=path, workspace=work).cpu().numpy().sum(0), want)
    finally:
        G.close()


def test_requests_of_few_sources_count_as_few():
    # four requests of one source are 128 packed columns, eight 256
    import torch
    for make, r, kernel, steps in ((lambda: gg.erdos_renyi(1 << 17, 64, weights=(1, 4), seed=18), 4, "dist_mfbr", True),
                                   (lambda: gg.erdos_renyi(60000, 9, seed=19), 8, "level_mfbf_gather", False)):
        g = make()
        srcs = gg.sample_sources(g, r, seed=20)
        G = mfbc.Graph.from_csr(g)
        try:
            lists = [torch.from_numpy(srcs[i:i + 1]).cuda() for i in range(r)]
            lam, prof = G.bc_multi(lists, profile=True)
            assert (kernel in prof["kernels"]) == steps
            # in the workspace that the columns ask for, whichever kernels that is for
            for n_b in (0, 32, 256):
                work = torch.empty(G.workspace_size(32 * r, 2, n_b=n_b), dtype=torch.uint8, device="cuda")
                close(G.bc_multi(lists, n_b=n_b, workspace=work).cpu().numpy(), lam.cpu().numpy())
            for i in range(r):
                close(lam[i].cpu().numpy(), oracle.bc(g, srcs[i:i + 1]))
        finally:
            G.close()
