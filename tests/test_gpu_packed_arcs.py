"""A weighted graph's second copy of its arcs (column and weight in one word, for
the source kernel): kept only where a call can run by source.
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


def test_arcs_are_packed_only_where_a_call_can_use_them():
    # weights past the distance families' 4096: no second copy of the arcs (4
    # bytes each, in both orientations), and the calls run as before
    import torch

    n, m = 1 << 16, 5_000_000
    rng = np.random.default_rng(5)
    key = np.unique(rng.integers(0, n, m) * n + rng.integers(0, n, m))
    key = key[key // n != key % n]
    rowptr = np.zeros(n + 1, np.int64)
    rowptr[1:] = np.cumsum(np.bincount(key // n, minlength=n))
    col = (key % n).astype(np.int32)
    held = {}
    for wmax in (100, 5000, 100, 5000):                 # (the first two also load modules and pools)
        w = rng.integers(1, wmax, len(key)).astype(np.int32)
        w[0] = wmax
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        G = mfbc.Graph(rowptr, col, w, directed=True)
        held[wmax] = before - torch.cuda.mem_get_info()[0]
        srcs = np.array([1, 77], np.int32)
        g = gg.CSRGraph(n=n, rowptr=rowptr, col=col, w=w, directed=True)
        if wmax == 5000:
            d, s = G.sssp(srcs)
            wd, ws, _ = oracle.sssp(g, srcs)
            assert np.array_equal(d, wd) and np.array_equal(s, ws)
            with pytest.raises(mfbc.MFBCError):
                G.bc(srcs, path=mfbc.PATH_DIST)
        G.close()
    assert held[100] - held[5000] >= 2 * 4 * len(key) - (4 << 20)
