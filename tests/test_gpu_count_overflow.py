"""Path counts that pass 2^64 in a single sum, through the C ABI against the
CPU oracle.

The unit-weight kernels keep sigma_bar in 64 bits and hand a source whose counts
reach 2^58 to kernels that count in FP64.  The counts here stay below 2^58 up to
the last layer but one, whose vertices then meet in one vertex: the sum is 2^64
(0 in 64 bits), or 2^64 plus one or two terms (again below 2^58 in 64 bits), so
that only the sum's own overflow shows it.  Few predecessors are summed by one
warp; more than 512 by the warps of a block in pieces.

Every count is a power of two times a small integer, exact in FP64: tau and
sigma_bar bit-exact, lambda within 1e-9 relative with exact zeros, and the
inexact-count warning (sigma_bar >= 2^53).
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


def funnel(layers, mids, n, directed):
    """Vertex 0, `layers` complete layers of 4 vertices, `mids` vertices joined to
    the last layer, one vertex joined to all of them, one behind it; isolated
    vertices up to n.  From 0, sigma_bar of the meeting vertex is mids * 4^layers."""
    edges = [(0, 1 + i) for i in range(4)]
    for k in range(layers - 1):
        edges += [(1 + 4 * k + i, 5 + 4 * k + j) for i in range(4) for j in range(4)]
    first = 1 + 4 * layers
    meet = first + mids
    edges += [(first - 4 + i, first + j) for i in range(4) for j in range(mids)]
    edges += [(first + j, meet) for j in range(mids)]
    edges += [(meet, meet + 1)]
    return gg.from_edges(max(n, meet + 2), edges, directed=directed)


# layers, predecessors of the meeting vertex: 2^64, 2^64 + 2^56, 2^64, 2^64 + 2^55
SHAPES = [(28, 256), (28, 257), (27, 1024), (27, 1026)]


# 9000 vertices: a graph of the level family, whose calls of few sources run by
# source too
@pytest.mark.parametrize("n", [0, 9000])
@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("layers,mids", SHAPES)
def test_a_sum_past_2p64_is_found(layers, mids, directed, n):
    import torch
    g = funnel(layers, mids, n, directed)
    meet = 1 + 4 * layers + mids
    srcs = np.array([0, 1, meet + 1, 0, 40], np.int32)
    want = oracle.bc(g, srcs)
    wd, ws, _ = oracle.sssp(g, srcs)
    assert ws[0, meet] == float(mids * 4**layers) >= 2.0**64
    G = mfbc.Graph.from_csr(g)
    try:
        for p in (mfbc.PATH_AUTO, mfbc.PATH_SMALL, mfbc.PATH_LEVEL):
            lam, warn = G.bc(srcs, path=p, return_warn=True)
            close(lam, want)
            assert warn & mfbc.MFBC_WARN_SIGMA_INEXACT
            d, s = G.sssp(srcs, path=p)
            assert np.array_equal(d, wd) and np.array_equal(s, ws)
            lists = [torch.from_numpy(x).cuda() for x in (srcs[:1], srcs[1:])]
            rows = G.bc_multi(lists, path=p).cpu().numpy()
            close(rows[0], oracle.bc(g, srcs[:1]))
            close(rows[1], oracle.bc(g, srcs[1:]))
    finally:
        G.close()
