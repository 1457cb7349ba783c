"""Graph construction on the device (row structure and arc checks) and the level
kernels' source-major rows, at the edges of their blocks: vertex counts around
the one from which the rows are built on the device and off a multiple of 32,
rows of no arcs, one item and several, arcs on both sides of a block of the
checks.  Bars: tau and sigma_bar bit-exact, lambda within 1e-9 relative with
exact zeros."""
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


def rows(n, directed, seed):
    """Rows of 0..5 arcs, a tenth empty, and 32 each of the lengths around an item's 32 arcs."""
    rng = np.random.default_rng(seed)
    deg = rng.integers(0, 6, n)
    deg[rng.integers(0, n, n // 10)] = 0
    deg[rng.choice(n, 32 * 7, replace=False)] = np.tile([31, 32, 33, 63, 64, 65, 1100], 32)
    deg[-1] = 0
    u = np.repeat(np.arange(n), deg)
    v = rng.integers(0, n, u.size)
    u, v = u[u != v], v[u != v]
    if not directed:
        u, v = np.concatenate([u, v]), np.concatenate([v, u])
    key = np.unique(u.astype(np.int64) * n + v)
    rp = np.zeros(n + 1, np.int64)
    np.add.at(rp, key // n + 1, 1)
    return gg.CSRGraph(n=n, rowptr=np.cumsum(rp), col=(key % n).astype(np.int32), w=None, directed=directed)


@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("n, k", [(8192, 40), (8193, 33), (9217, 130), (33000, 1)])
def test_level_kernels_on_built_rows(n, k, directed):
    g = rows(n, directed, n + directed)
    srcs = gg.sample_sources(g, k, seed=1)
    G = mfbc.Graph.from_csr(g)
    lam = G.bc(srcs, path=mfbc.PATH_LEVEL)
    want = oracle.bc(g, srcs)
    zero = want == 0
    assert np.array_equal(lam[zero], want[zero])
    assert np.all(np.abs(lam[~zero] - want[~zero]) <= 1e-9 * want[~zero])
    d, s = G.sssp(srcs, path=mfbc.PATH_LEVEL)
    wd, ws, _ = oracle.sssp(g, srcs)
    assert np.array_equal(d, wd) and np.array_equal(s, ws)
    G.close()


def without(g, k):
    """g (and its weights) without arc k."""
    rp = g.rowptr.copy()
    rp[np.searchsorted(g.rowptr, k, side="right"):] -= 1
    return rp, np.delete(g.col, k), None if g.w is None else np.delete(g.w, k)


@pytest.mark.parametrize("weights", [None, (1, 9)])
def test_every_arc_is_checked(weights):
    # hub 0 with 3000 leaves (arcs of one row over several blocks), leaves joined at random
    rng = np.random.default_rng(7)
    n = 3100
    u = np.concatenate([np.zeros(3000, np.int64), rng.integers(1, n, 4000)])
    v = np.concatenate([np.arange(1, 3001), rng.integers(1, n, 4000)])
    u, v = u[u != v], v[u != v]
    lo, hi = np.minimum(u, v), np.maximum(u, v)
    key = np.unique(lo * n + hi)
    w = None if weights is None else rng.integers(weights[0], weights[1] + 1, key.size)
    both = np.concatenate([key, key % n * n + key // n])
    order = np.argsort(both)
    rp = np.zeros(n + 1, np.int64)
    np.add.at(rp, both // n + 1, 1)
    g = gg.CSRGraph(n=n, rowptr=np.cumsum(rp), col=(both[order] % n).astype(np.int32),
                    w=None if w is None else np.tile(w, 2)[order].astype(np.int32), directed=False)
    mfbc.Graph(g.rowptr, g.col, g.w, directed=False).close()
    nnz = g.col.size
    for k in (0, 1023, 1024, 2999, 3000, 3001, nnz // 2, nnz - 1):
        bad = [without(g, k)]
        if g.w is not None:
            changed = g.w.copy()
            changed[k] += 1
            bad.append((g.rowptr, g.col, changed))
        for a in bad:
            with pytest.raises(mfbc.MFBCError) as e:
                mfbc.Graph(*a, directed=False)
            assert e.value.status == mfbc.MFBC_ERR_INVALID and "symmetric" in str(e.value)
        # of an arc that has no reverse, in a directed graph, nothing is asked
        mfbc.Graph(*bad[0], directed=True).close()
        for value, word in ((n, "range"), (-1, "range"), (int(np.searchsorted(g.rowptr, k, side="right")) - 1, "self-loop")):
            col = g.col.copy()
            col[k] = value
            with pytest.raises(mfbc.MFBCError, match=word):
                mfbc.Graph(g.rowptr, col, g.w, directed=False)
        if k:
            col = g.col.copy()
            col[k] = col[k - 1]
            if g.rowptr[np.searchsorted(g.rowptr, k, side="right") - 1] < k:     # not a row's first arc
                with pytest.raises(mfbc.MFBCError, match="sorted"):
                    mfbc.Graph(g.rowptr, col, g.w, directed=False)
