"""The sweep's lane shapes: the half-lane ones (two chunks to a lane), which a handle has only after the
autotuner picked one, at every row class's borders, and both kinds on batches of tiny graphs."""
import functools

import numpy as np
import pytest

import oracle
import peek
from paper_1601_05527_gb300 import graphgen
from gpu_util import assert_rho_close, entry_weights_f64, lib, rho_error
from test_gpu_row_teams import border_graph, distances

pytestmark = pytest.mark.gpu

STORAGE = {"fp32": 4, "bf16": 8, "fp16": 8, "q16": 8}   # values to a 16-byte chunk


def natural_lanes(storage, R):
    chunks = -(-R // STORAGE[storage])
    return 1 << (chunks - 1).bit_length()


@functools.lru_cache(None)
def reference(R, weighted):
    g = border_graph(weighted)
    return oracle.algebraic_distance(g.row_ptr, g.col, entry_weights_f64(g), R=R, k=7, omega=0.5, seed=11)


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("R", [8, 13, 16, 32, 50, 64, 128, 250])
@pytest.mark.parametrize("storage", list(STORAGE))
def test_half_lane_shape(storage, R, weighted):
    lanes = natural_lanes(storage, R)
    if not 2 <= lanes <= 32:
        pytest.skip("one chunk to a row, or two to a lane already")
    L = lib()
    g = border_graph(weighted)
    h = L.ad_graph_create(g.n, g.row_ptr, g.col, g.weight)
    natural = distances(L, h, g.m, R, storage)
    at32 = distances(L, h, g.m, 32, storage)
    peek.set_shape(h, R, L.STORAGES[storage], lanes // 2, 2)
    rho = distances(L, h, g.m, R, storage)
    L.ad_graph_destroy(h)
    ref = reference(R, weighted)
    if storage == "fp32":
        assert_rho_close(rho, ref)
    else:   # the vectors are rounded independently of one another: any number of them errs about as 32 do
        bound = 4 * rho_error(at32, reference(32, weighted)) * max(1.0, (32 / R) ** 0.5)
        assert rho_error(natural, ref) <= bound
        assert rho_error(rho, ref) <= bound


@pytest.mark.parametrize("half", [False, True])
@pytest.mark.parametrize("R", [1, 7, 33, 64, 130, 250])
@pytest.mark.parametrize("storage", list(STORAGE))
def test_batch_of_tiny_graphs(storage, R, half):
    lanes = natural_lanes(storage, R)
    if half and not 2 <= lanes <= 32:
        pytest.skip("one chunk to a row, or two to a lane already")
    L = lib()
    dot = graphgen.from_edges(1, np.zeros(0, np.int64), np.zeros(0, np.int64))
    pair = graphgen.from_edges(2, [0], [1])
    graphs = [pair, dot, graphgen.grid2d(2, 2), graphgen.watts_strogatz(20, 4, 0.2, seed=1), dot, pair, pair,
              graphgen.watts_strogatz(33, 6, 0.2, seed=2), graphgen.rmat(9, 20, seed=3), graphgen.grid2d(3, 5)] * 3
    voff, big = graphgen.concat(graphs)
    h = L.ad_graph_create_batched(voff, big.n, big.row_ptr, big.col, None)
    if half:
        peek.set_shape(h, R, L.STORAGES[storage], lanes // 2, 2)
    rho = distances(L, h, big.m, R, storage)
    at = L.ad_graph_edge_offsets(h)
    L.ad_graph_destroy(h)
    for k, g in enumerate(graphs):
        if g.m == 0:
            continue
        h = L.ad_graph_create(g.n, g.row_ptr, g.col, None)
        if half:
            peek.set_shape(h, R, L.STORAGES[storage], lanes // 2, 2)
        assert np.array_equal(rho[at[k]:at[k + 1]], distances(L, h, g.m, R, storage)), k
        L.ad_graph_destroy(h)
