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
