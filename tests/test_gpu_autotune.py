"""The autotuner times every launch shape once: no candidate that comes to the same grid as another."""
import pytest

from paper_1601_05527_gb300 import graphgen
from gpu_util import lib

pytestmark = pytest.mark.gpu

RUN = 6   # launches of a run: start vectors, four sweeps, distances


@pytest.mark.parametrize("storage,R,grids", [("fp32", 32, 1), ("fp32", 8, 1), ("fp16", 32, 2), ("bf16", 64, 2), ("q16", 32, 2)])
def test_no_equal_candidates(storage, R, grids):
    # FP32 sweeps fit four CTAs on an SM (64 registers a thread), 16-bit ones five (48): 5 and 4 of the
    # candidates are the full grid again, or 5 is
    L, g = lib(), graphgen.rmat(12, 16, seed=4)
    h = L.ad_graph_create(g.n, g.row_ptr, g.col, None)
    L.ad_graph_autotune(h, R, storage)   # the plans of both shapes
    before = L.ad_kernel_launch_count()
    L.ad_graph_autotune(h, R, storage)
    L.ad_graph_destroy(h)
    assert L.ad_kernel_launch_count() - before == 2 * grids * 3 * RUN   # two lane shapes, three runs each
