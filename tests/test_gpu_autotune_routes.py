"""A tuned handle against an untuned one: tuning must not take away the kernels
that AUTO would have run faster.

  * unit-weight graph past the small family's sizes: only the level kernels are
    timed, and calls of few sources still run one block per source;
  * unit-weight graph of both families: where the level kernels won for the
    tuned number of sources they keep it, with fewer the source kernel may run;
  * small family: every width runs the same kernel, so none is kept as a cap;
  * weighted graph tuned within the general family: AUTO still runs by source.
Results against the CPU oracle, lambda within 1e-9 relative with exact zeros.
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


def run(G, g, srcs):
    lam, prof = G.bc(srcs, profile=True)
    want = oracle.bc(g, srcs)
    assert np.array_equal(lam == 0, want == 0)
    assert np.max(np.abs(lam - want)[want != 0] / want[want != 0]) <= 1e-9
    return prof


def test_level_family_keeps_the_source_kernel_for_few_sources():
    g = gg.erdos_renyi(60000, 8, seed=1)
    srcs = gg.sample_sources(g, 600, seed=2)
    G = mfbc.Graph.from_csr(g)
    assert G.autotune(srcs)["path"] == mfbc.PATH_LEVEL
    assert "level_mfbf_gather" not in run(G, g, srcs[:64])["kernels"]
    assert "level_mfbf_gather" in run(G, g, srcs)["kernels"]
    G.close()


def test_level_family_tuned_against_the_small_one():
    g = gg.rmat(14, 16, seed=3)
    srcs = gg.sample_sources(g, 3000, seed=4)          # the level kernels win by 1.5
    G = mfbc.Graph.from_csr(g)
    assert G.autotune(srcs)["path"] == mfbc.PATH_LEVEL
    assert "level_mfbf_gather" in run(G, g, srcs)["kernels"]
    assert "level_mfbf_gather" not in run(G, g, srcs[:64])["kernels"]
    # a family tuned alone: the same choice
    G.close()
    G = mfbc.Graph.from_csr(g)
    G.autotune(srcs[:512], path=mfbc.PATH_LEVEL)
    assert "level_mfbf_gather" not in run(G, g, srcs[:64])["kernels"]
    G.close()


def test_small_family_keeps_no_width():
    g = gg.rmat(11, 8, seed=5)
    srcs = gg.sample_sources(g, 700, seed=6)
    G = mfbc.Graph.from_csr(g)
    t = G.autotune(srcs, path=mfbc.PATH_SMALL)
    assert t["n_b"] == 256 and t["tried"] == 4
    d, s, prof = G.sssp(srcs, profile=True)
    assert prof["n_b"] >= 700                          # rows staged in one piece
    wd, ws, _ = oracle.sssp(g, srcs)
    assert np.array_equal(d, wd) and np.array_equal(s, ws)
    G.close()


def test_general_family_tuned_alone_leaves_auto_by_source():
    g = gg.rmat(12, 8, weights=(1, 255), directed=True, seed=7)
    srcs = gg.sample_sources(g, 200, seed=8)
    G = mfbc.Graph.from_csr(g)
    G.autotune(srcs, path=mfbc.PATH_GENERAL)
    prof = run(G, g, srcs)
    assert prof["path"] == mfbc.PATH_GENERAL and "mfbf_accumulate" not in prof["kernels"]
    lam, prof = G.bc(srcs, path=mfbc.PATH_GENERAL, profile=True)
    assert "mfbf_accumulate" in prof["kernels"]
    G.close()
