"""The exponent search on batches with far more graphs than edges."""
import numpy as np
import pytest

import oracle
from paper_1601_05527_gb300 import graphgen
from gpu_util import lib
from test_gpu_fit_known import GRAPHS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["local", "global"])
@pytest.mark.parametrize("fraction", [0.25, 0.5, 0.9])
def test_more_graphs_than_edges(fraction, mode):
    # the few graphs with edges lie far apart among 1,500 of one vertex each: more problems than
    # a launch sized by the edges has threads
    L = lib()
    dot = graphgen.from_edges(1, np.zeros(0, np.int64), np.zeros(0, np.int64))
    graphs = [dot] * 1500
    for at, name in zip([3, 300, 700, 1400, 1499], ["star", "edge", "grid", "ring4", "rmat"]):
        graphs[at] = GRAPHS[name]()
    voff, big = graphgen.concat(graphs)
    score = graphgen.random_scores(big.m, n_distinct=max(2, big.m // 3), seed=4)
    h = L.ad_graph_create_batched(voff, big.n, big.row_ptr, big.col, None)
    keep = np.zeros(big.m, np.uint8)
    L.ad_sparsify_scores(h, score, fraction, mode, "per_node", keep)
    at = L.ad_graph_edge_offsets(h)
    L.ad_graph_destroy(h)
    for k, g in enumerate(graphs):
        if g.m:
            s = score[at[k]:at[k + 1]].astype(np.float64)
            ref, _, _ = oracle.sparsify(g.row_ptr, g.col, s, mode, "per_node", fraction)
            assert np.array_equal(keep[at[k]:at[k + 1]], ref), k
