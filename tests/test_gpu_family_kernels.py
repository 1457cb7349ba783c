"""The kernels of the small and distance families themselves (small.cu, dist.cu),
through the C ABI against the CPU oracle.

Most calls of these families run one block per source (source.cu); the
MFBC_OPT_TEST_FAMILY_KERNELS hook gives them to the family's own kernels, which
take what the source kernel does not: few sources of large weighted graphs, and
graphs and workspaces that it cannot hold.

  * persistent small-graph kernel: its queue of batches with a ragged last one,
    packed requests, MFBF rows, and the batches it hands to the general kernels
    (counts of 2^58 and more, also where one sum passes 2^64; deeper than 254 levels);
  * distance step kernels: weights with gaps (five flag words an item), ragged
    batches, a hub, the one-item scan of dense graphs, repeated sources, packed
    requests, and batches of 1024 and 4096 columns.

Bars: tau and sigma_bar bit-exact below 2^53, lambda within 1e-9 relative with
exact zeros.
"""
import numpy as np
import pytest

import graphgen as gg
import oracle
import paper_1609_07008_gb300 as mfbc

pytestmark = pytest.mark.gpu
SMALL, DIST = mfbc.PATH_SMALL, mfbc.PATH_DIST


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


def check(g, srcs, path, n_b, rows=50, sigma=True):
    """bc, sssp and bc_multi of the family's kernels; returns bc's profile and warnings."""
    import torch
    G = mfbc.Graph.from_csr(g)
    kw = dict(n_b=n_b, path=path, test_family_kernels=True)
    try:
        lam, warn, prof = G.bc(srcs, return_warn=True, profile=True, **kw)
        close(lam, oracle.bc(g, srcs))
        if path == DIST:                 # (MFBr of the source kernel is part of its one launch)
            assert prof["kernels"]["dist_mfbr"]["launches"] > 0
        if sigma:
            d, s = G.sssp(srcs[:rows], **kw)
            wd, ws, _ = oracle.sssp(g, srcs[:rows])
            assert np.array_equal(d, wd) and np.array_equal(s, ws)
        cut = max(1, len(srcs) // 3)
        lists = [srcs[:cut], srcs[cut:], srcs[:1]]
        lam = G.bc_multi([torch.from_numpy(x).cuda() for x in lists], **kw).cpu().numpy()
        for r, x in enumerate(lists):
            close(lam[r], oracle.bc(g, x))
        return prof, warn
    finally:
        G.close()


@pytest.mark.parametrize("n_b", [32, 64, 128, 256])
def test_small_queue_of_batches(n_b):
    g = gg.rmat(12, 8, seed=3)
    srcs = gg.sample_sources(g, 1000, seed=4)          # ragged for every width
    prof, _ = check(g, srcs, SMALL, n_b)
    assert prof["batches"] == prof["fwd_iters"] == -(-1000 // n_b)   # (the source kernel counts steps)


def test_small_directed_with_unreachable_pairs():
    g = gg.rmat(11, 8, directed=True, seed=5)
    check(g, gg.sample_sources(g, 300, seed=6), SMALL, 64)


def grid(L):
    edges = [(r * L + c, r * L + c + 1) for r in range(L) for c in range(L - 1)]
    edges += [(r * L + c, (r + 1) * L + c) for r in range(L - 1) for c in range(L)]
    return gg.from_edges(L * L, edges, directed=False)


def test_small_counts_past_2p58_are_redone():
    corners = np.array([0, 39, 40 * 39, 40 * 40 - 1, 20 * 40 + 20], np.int32)
    _, warn = check(grid(40), corners, SMALL, 32, sigma=False)
    assert warn & mfbc.MFBC_WARN_SIGMA_INEXACT


def test_small_sum_past_2p64_is_redone():
    # 28 layers of 4, then 256 vertices of 2^56 paths each that meet in one
    layers, mids = 28, 256
    first = 1 + 4 * layers
    e = [(0, 1 + i) for i in range(4)]
    e += [(1 + 4 * k + i, 5 + 4 * k + j) for k in range(layers - 1) for i in range(4) for j in range(4)]
    e += [(first - 4 + i, first + j) for i in range(4) for j in range(mids)]
    e += [(first + j, first + mids) for j in range(mids)] + [(first + mids, first + mids + 1)]
    g = gg.from_edges(first + mids + 2, e, directed=True)
    _, warn = check(g, np.array([0, 1, 0], np.int32), SMALL, 32)      # (every count is exact in FP64)
    assert warn & mfbc.MFBC_WARN_SIGMA_INEXACT


def test_small_deeper_than_byte_levels_is_redone():
    n = 700
    g = gg.from_edges(n, [(i, i + 1) for i in range(n - 1)], directed=False)
    check(g, np.array([0, 1, 350, 699, 5, 5], np.int32), SMALL, 32)


def weighted(n, deg, weights, seed):
    rng = np.random.default_rng(seed)
    u, v = rng.integers(0, n, (2, n * deg))
    keep = u != v
    w = rng.choice(np.asarray(weights), n * deg)
    return gg.from_edges(n, list(zip(u[keep].tolist(), v[keep].tolist())), directed=True, weights=w[keep].tolist())


def hub(n, seed):
    rng = np.random.default_rng(seed)
    edges = [(0, v) for v in range(1, n)]
    edges += [(int(a), int(b)) for a, b in rng.integers(1, n, (3000, 2)) if a != b]
    return gg.from_edges(n, edges, directed=False, weights=rng.integers(1, 6, len(edges)).tolist())


DIST_CASES = {
    "weight_gaps": (lambda: weighted(3000, 6, [1, 40, 77, 128], 11), 100, 64),
    "ragged_words": (lambda: gg.grid2d(24, weights=(1, 16), seed=4), 45, 32),
    "hub": (lambda: hub(2000, 7), 70, 0),
    "one_item_scan": (lambda: gg.erdos_renyi(2000, 40, weights=(1, 10), seed=9), 96, 0),
    "unit_weights_directed": (lambda: gg.rmat(11, 8, directed=True, seed=11), 130, 128),
}


@pytest.mark.parametrize("name", DIST_CASES)
def test_dist_steps(name):
    make, k, n_b = DIST_CASES[name]
    g = make()
    check(g, gg.sample_sources(g, k, seed=3), DIST, n_b)


def test_dist_steps_repeated_sources():
    check(gg.grid2d(16, weights=(1, 16), seed=12), np.array([5, 77, 5, 5, 77], np.int32), DIST, 0)


@pytest.mark.parametrize("n_b", [1024, 4096])
def test_dist_steps_wide_batches(n_b):
    g = gg.grid2d(64, weights=(1, 16), seed=1)
    prof, _ = check(g, gg.sample_sources(g, 4000, seed=2), DIST, n_b)
    assert prof["n_b"] == n_b


def test_general_and_level_families_under_auto():
    # AUTO runs these by source; with the hook their family's kernels do
    for g, kernel in ((gg.rmat(13, 8, weights=(1, 255), seed=6), "mfbf_pull"),
                      (gg.erdos_renyi(9000, 6, seed=7), "level_mfbf_gather")):
        srcs = gg.sample_sources(g, 40, seed=8)
        G = mfbc.Graph.from_csr(g)
        lam, prof = G.bc(srcs, profile=True, test_family_kernels=True)
        close(lam, oracle.bc(g, srcs))
        assert prof["kernels"][kernel]["launches"] > 0
        lam, prof = G.bc(srcs, profile=True)
        close(lam, oracle.bc(g, srcs))
        assert kernel not in prof["kernels"]
        G.close()
