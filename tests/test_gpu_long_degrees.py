"""Weighted degrees of rows that a block sums (above 2,048 entries), bit for bit: parallel sums where
they are exact in any order, CSR order otherwise."""
import numpy as np
import pytest

import peek
from paper_1601_05527_gb300 import graphgen
from gpu_util import lib

pytestmark = pytest.mark.gpu

DEGREES = [2047, 2048, 2049, 2049, 4096, 4097, 6144, 10000]
POOL = 10100


def hubs():
    rng = np.random.default_rng(1)
    H = len(DEGREES)
    u = np.repeat(np.arange(H), DEGREES)
    v = np.concatenate([H + rng.choice(POOL, d, replace=False) for d in DEGREES])
    return graphgen.from_edges(H + POOL, u, v)


def weights(g, kind, seed):
    """narrow: 11 bits of mantissa over two binary orders, exact; wide: full mantissas over 40 orders;
    mixed: every other hub wide."""
    rng = np.random.default_rng(seed)
    narrow = (1 + rng.integers(0, 2048, g.m) / 2048) * 2.0 ** rng.integers(0, 2, g.m)
    wide = rng.uniform(1, 2, g.m) * 2.0 ** rng.integers(-20, 21, g.m)
    pick = {"narrow": np.zeros(g.m, bool), "wide": np.ones(g.m, bool), "mixed": edge_hub(g) % 2 == 1}[kind]
    return np.where(pick, wide, narrow).astype(np.float32)


def edge_hub(g):
    """Smaller end of every edge, in edge order (by smaller end, then larger end)."""
    row = np.repeat(np.arange(g.n), np.diff(g.row_ptr))
    return row[g.col > row]


def expected(g, w):
    """Sums in CSR order and the exactness rule: all partial sums fit 53 bits."""
    D, exact = np.zeros(g.n), np.zeros(g.n, np.uint8)
    for i in range(g.n):
        x = w[g.row_ptr[i]:g.row_ptr[i + 1]]
        D[i] = np.add.accumulate(x.astype(np.float64))[-1] if len(x) else 0.0
        e = (x.view(np.uint32) >> 23) & 0xff
        exact[i] = len(x) == 0 or int(e.max()) - max(int(e.min()), 1) + int(np.ceil(np.log2(len(x)))) + 24 <= 53
    return D, exact


@pytest.mark.parametrize("kind", ["narrow", "wide", "mixed"])
def test_degrees_bit_for_bit(kind):
    L, g0 = lib(), hubs()
    g = graphgen.with_edge_weights(g0, weights(g0, kind, 2))
    h = L.ad_graph_create(g.n, g.row_ptr, g.col, g.weight)
    for seed in (None, 3, 4):
        if seed is not None:
            w_edge = weights(g0, kind, seed)
            g = graphgen.with_edge_weights(g0, w_edge)
            L.ad_graph_set_edge_weights(h, w_edge)
        D, exact = peek.degrees(h, g.n)
        ref, ref_exact = expected(g, g.weight)
        assert np.array_equal(D.view(np.uint64), ref.view(np.uint64))
        assert np.array_equal(exact, ref_exact)
        wide_hubs = {"narrow": 0, "wide": len(DEGREES), "mixed": len(DEGREES) // 2}[kind]
        assert (exact[:len(DEGREES)] == 0).sum() == wide_hubs
    L.ad_graph_destroy(h)


def test_weight_update_allocates_no_list():
    import torch
    L, g0 = lib(), hubs()
    w = torch.from_numpy(weights(g0, "wide", 5)).cuda()
    h = L.ad_graph_create(g0.n, g0.row_ptr, g0.col, None)
    L.ad_graph_set_edge_weights(h, w)
    torch.cuda.synchronize()
    before = torch.cuda.memory_stats()["allocation.all.allocated"]
    L.ad_graph_set_edge_weights(h, w)
    torch.cuda.synchronize()
    # the first bad weight's place, the counts of upper entries, the largest degree of each graph
    assert torch.cuda.memory_stats()["allocation.all.allocated"] - before <= 3
    L.ad_graph_destroy(h)
