"""The profile's label of the one-block-per-source kernel in each family (mfbc.h,
mfbc_kernel_stat): calls of the level and general families that it takes do not
appear under kernels of other families."""
import pytest

import graphgen as gg
import paper_1609_07008_gb300 as mfbc

pytestmark = pytest.mark.gpu

CASES = {
    "level": (lambda: gg.erdos_renyi(9000, 6, seed=1), mfbc.PATH_LEVEL, "source_bc"),
    "general": (lambda: gg.rmat(12, 8, weights=(1, 255), seed=2), mfbc.PATH_GENERAL, "source_bc"),
    "small": (lambda: gg.rmat(11, 8, seed=3), mfbc.PATH_SMALL, "small_persistent"),
    "dist": (lambda: gg.grid2d(30, weights=(1, 9), seed=4), mfbc.PATH_DIST, "dist_mfbf"),
}


@pytest.mark.parametrize("name", CASES)
def test_label_of_the_source_kernel(name):
    from paper_1609_07008_gb300 import build
    build.build()
    make, path, label = CASES[name]
    g = make()
    with mfbc.Graph.from_csr(g) as G:
        _, prof = G.bc(gg.sample_sources(g, 20, seed=5), profile=True, count_bytes=True)
    assert prof["path"] == path
    k = prof["kernels"][label]
    assert k["launches"] == 1 and k["ms"] > 0 and k["bytes"] > 0
    others = {"small_persistent", "dist_mfbf", "dist_mfbr", "source_bc", "level_mfbf_gather", "mfbf_accumulate"} - {label}
    assert not others & set(prof["kernels"])
