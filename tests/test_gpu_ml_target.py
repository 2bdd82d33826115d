"""The shared ratio that reaches a target fraction: the smallest grid point that does, whatever levels
are sparsified (the search counts at the finest of them, without going down to the input graph)."""
import numpy as np
import pytest

import oracle
from paper_1601_05527_gb300 import graphgen
from gpu_util import lib

pytestmark = pytest.mark.gpu

STEP = 2.0 ** -20


@pytest.mark.parametrize("levels", ["coarse", "fine", "whole", "coarsest", "finest", "none"])
@pytest.mark.parametrize("weighted", [False, True])
def test_ratio_is_the_smallest(levels, weighted):
    L = lib()
    g = graphgen.barabasi_albert(6000, 6, seed=3)
    if weighted:
        g = graphgen.with_edge_weights(g, graphgen.lognormal_edge_weights(g.m, seed=4))
    h = L.ad_graph_create(g.n, g.row_ptr, g.col, g.weight)
    ml = L.ad_ml_build(h, R=8, k=10, omega=0.5, seed=5, Q=0.5, coarsest_n=200, mode="local")
    n = L.ad_ml_levels(ml)
    assert n >= 3
    span = max(1, n // 2)
    pick = {"coarse": range(span), "fine": range(n - span, n), "whole": range(n), "coarsest": [0], "finest": [n - 1],
            "none": []}[levels]   # ratio l belongs to the l-th coarsest level

    def ratios(r):
        x = -np.ones(n)
        x[list(pick)] = r
        return x

    keep = np.zeros(g.m, np.uint8)
    low, _ = L.ad_ml_sparsify(ml, ratios(0.0), -1.0, keep)   # the coarsest levels alone cannot go below this
    for share in (0.05, 0.5, 0.95):
        K = low + int(share * (g.m - low))
        kept, r = L.ad_ml_sparsify(ml, ratios(1.0), K / g.m, keep)
        K = oracle.target_count(g.m, K / g.m)
        assert kept == keep.sum() >= K
        at_r = np.zeros(g.m, np.uint8)
        assert L.ad_ml_sparsify(ml, ratios(r), -1.0, at_r)[0] == kept and np.array_equal(at_r, keep)
        if r > STEP:
            assert L.ad_ml_sparsify(ml, ratios(r - STEP), -1.0, at_r)[0] == at_r.sum() < K
    L.ad_ml_destroy(ml)
    L.ad_graph_destroy(h)
