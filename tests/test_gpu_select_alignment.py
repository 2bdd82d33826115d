"""Whole-graph selection on device arrays that start anywhere: the vector and the
scalar form of its passes, tile remainders, ties at the threshold."""
import numpy as np
import pytest

import oracle
from paper_1601_05527_gb300 import graphgen
from gpu_util import lib

pytestmark = pytest.mark.gpu


def path_graph(m):
    return graphgen.from_edges(m + 1, np.arange(m), np.arange(1, m + 1))


@pytest.mark.parametrize("mode", ["local", "global"])
@pytest.mark.parametrize("score_off,keep_off", [(0, 0), (1, 0), (0, 3), (2, 5), (4, 16)])
@pytest.mark.parametrize("m", [1, 15, 16, 17, 4095, 4096, 4097, 4112, 12289])
def test_offsets(m, score_off, keep_off, mode):
    import torch
    L, g = lib(), path_graph(m)
    score = graphgen.random_scores(m, n_distinct=max(1, m // 50), seed=m)
    sd = torch.zeros(m + 8, device="cuda")
    sd[score_off:score_off + m] = torch.from_numpy(score)
    kd = torch.full((m + 32,), 7, dtype=torch.uint8, device="cuda")
    view = kd[keep_off:keep_off + m]
    h = L.ad_graph_create(g.n, g.row_ptr, g.col, None)
    for fraction in (0.0, 0.37, 1.0):
        kept, _ = L.ad_sparsify_scores(h, sd[score_off:score_off + m], fraction, mode, "whole_graph", view)
        torch.cuda.synchronize()
        ref, ref_kept, _ = oracle.sparsify(g.row_ptr, g.col, score.astype(np.float64), mode, "whole_graph", fraction)
        got = kd.cpu().numpy()
        assert kept == ref_kept
        assert np.array_equal(got[keep_off:keep_off + m], ref)
        assert (got[:keep_off] == 7).all() and (got[keep_off + m:] == 7).all()
    L.ad_graph_destroy(h)


def test_batch_tiles_start_anywhere():
    L = lib()
    graphs = [path_graph(m) for m in (3, 4097, 1, 8191, 4096, 5)]
    voff, big = graphgen.concat(graphs)
    score = graphgen.random_scores(big.m, n_distinct=40, seed=9)
    h = L.ad_graph_create_batched(voff, big.n, big.row_ptr, big.col, None)
    at = L.ad_graph_edge_offsets(h)
    keep = np.zeros(big.m, np.uint8)
    L.ad_sparsify_scores(h, score, 0.3, "local", "whole_graph", keep)
    L.ad_graph_destroy(h)
    for k, g in enumerate(graphs):
        ref, _, _ = oracle.sparsify(g.row_ptr, g.col, score[at[k]:at[k + 1]].astype(np.float64), "local", "whole_graph", 0.3)
        assert np.array_equal(keep[at[k]:at[k + 1]], ref), k
