"""The sweep's row classes at their borders: rows of every degree at which the
work of a row changes hands (lane group, team of lanes, whole warp, chunks),
against the FP64 oracle, and a batch against its graphs one by one."""
import numpy as np
import pytest

import oracle
from paper_1601_05527_gb300 import graphgen
from gpu_util import assert_rho_close, entry_weights_f64, lib

pytestmark = pytest.mark.gpu

DEGREES = [1, 2, 3, 4, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 96, 127, 128, 129, 160, 511, 512, 513, 1024, 1025, 1537]


def border_graph(weighted, copies=3, seed=5):
    """`copies` vertices of each degree in DEGREES, joined to random vertices of a pool."""
    rng = np.random.default_rng(seed)
    hubs = np.repeat(DEGREES, copies)
    pool = 2100
    u = np.repeat(np.arange(len(hubs)), hubs)
    v = np.concatenate([len(hubs) + rng.choice(pool, d, replace=False) for d in hubs])
    g = graphgen.from_edges(len(hubs) + pool, u, v, name="borders")
    return graphgen.with_edge_weights(g, graphgen.lognormal_edge_weights(g.m, seed=seed)) if weighted else g


def distances(L, h, m, R, storage, flags=0):
    rho = np.zeros(m, np.float32)
    L.ad_algebraic_distance(h, R, 7, 0.5, 11, 0, storage, flags, rho)
    return rho


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("R", [2, 4, 7, 10, 16, 32, 50, 64, 130, 256])
def test_degree_borders_match_oracle(R, weighted):
    L = lib()
    g = border_graph(weighted)
    h = L.ad_graph_create(g.n, g.row_ptr, g.col, g.weight)
    rho = distances(L, h, g.m, R, "fp32")
    again = distances(L, h, g.m, R, "fp32", L.AD_DIST_PERSISTENT)
    L.ad_graph_destroy(h)
    ref = oracle.algebraic_distance(g.row_ptr, g.col, entry_weights_f64(g), R=R, k=7, omega=0.5, seed=11)
    assert_rho_close(rho, ref)
    assert np.array_equal(rho, again)


@pytest.mark.parametrize("storage", ["fp32", "bf16", "fp16", "q16"])
@pytest.mark.parametrize("R", [4, 16, 40])
def test_batch_equals_its_graphs(R, storage):
    # graphs of very different sizes, so that graphs meet inside one warp; the sums' order and the
    # bounds of the rescale do not depend on the neighbours in the batch: the same bits
    L = lib()
    graphs = [graphgen.watts_strogatz(n, 6, 0.2, seed=n) for n in (7, 9, 40, 8, 701)]
    graphs += [border_graph(False, copies=2), graphgen.grid2d(3, 3), border_graph(False, copies=1, seed=6)]
    voff, big = graphgen.concat(graphs)
    h = L.ad_graph_create_batched(voff, big.n, big.row_ptr, big.col, None)
    rho = distances(L, h, big.m, R, storage)
    at = L.ad_graph_edge_offsets(h)
    L.ad_graph_destroy(h)
    for k, g in enumerate(graphs):
        h = L.ad_graph_create(g.n, g.row_ptr, g.col, None)
        assert np.array_equal(rho[at[k]:at[k + 1]], distances(L, h, g.m, R, storage)), k
        L.ad_graph_destroy(h)
