"""The exponent search where few degrees share their breakpoints: passes whose
outcome follows from the tables alone, fractions below and above what one edge per
node keeps, batches whose graphs leave the search at different passes."""
import numpy as np
import pytest

import oracle
from paper_1601_05527_gb300 import graphgen
from gpu_util import lib

pytestmark = pytest.mark.gpu

FRACTIONS = [0.0, 0.05, 0.25, 0.4, 0.5, 0.75, 0.9, 1.0]


def star(n):
    return graphgen.from_edges(n, np.zeros(n - 1, np.int64), np.arange(1, n))


GRAPHS = {
    "ring4": lambda: graphgen.watts_strogatz(300, 4, 0.0, seed=1),      # one degree
    "ring10": lambda: graphgen.watts_strogatz(1000, 10, 0.1, seed=2),
    "grid": lambda: graphgen.grid2d(17, 23),
    "star": lambda: star(200),
    "rmat": lambda: graphgen.rmat(9, 8, seed=3),
    "edge": lambda: graphgen.from_edges(2, [0], [1]),
}


@pytest.mark.parametrize("mode", ["local", "global"])
@pytest.mark.parametrize("fraction", FRACTIONS)
@pytest.mark.parametrize("name", list(GRAPHS))
def test_single_graph(name, fraction, mode):
    L, g = lib(), GRAPHS[name]()
    score = graphgen.random_scores(g.m, n_distinct=max(2, g.m // 3), seed=4)
    h = L.ad_graph_create(g.n, g.row_ptr, g.col, None)
    keep = np.zeros(g.m, np.uint8)
    kept, e = L.ad_sparsify_scores(h, score, fraction, mode, "per_node", keep)
    L.ad_graph_destroy(h)
    ref, ref_kept, ref_e = oracle.sparsify(g.row_ptr, g.col, score.astype(np.float64), mode, "per_node", fraction)
    assert (kept, e) == (ref_kept, ref_e)
    assert np.array_equal(keep, ref)


@pytest.mark.parametrize("fraction", FRACTIONS)
def test_batch_of_unlike_graphs(fraction):
    L = lib()
    graphs = [make() for make in GRAPHS.values()] * 3
    voff, big = graphgen.concat(graphs)
    score = graphgen.random_scores(big.m, seed=5)
    h = L.ad_graph_create_batched(voff, big.n, big.row_ptr, big.col, None)
    at = L.ad_graph_edge_offsets(h)
    keep = np.zeros(big.m, np.uint8)
    L.ad_sparsify_scores(h, score, fraction, "global", "per_node", keep)
    L.ad_graph_destroy(h)
    for k, g in enumerate(graphs):
        ref, _, _ = oracle.sparsify(g.row_ptr, g.col, score[at[k]:at[k + 1]].astype(np.float64), "global", "per_node",
                                    fraction)
        assert np.array_equal(keep[at[k]:at[k + 1]], ref), k
