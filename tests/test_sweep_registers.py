"""Registers of the sweep kernels on 16-bit storage: at no lane shape may the rows in flight and the
partial sums of a lane outgrow the register bound.  Read off ptxas, so no GPU is needed."""
import os
import re
import subprocess

import pytest

from paper_1601_05527_gb300 import build

# (storage, lanes per row, chunks per lane): R = 33 .. 64 and 129 .. 256, and a shape only the autotuner takes
SHAPES = [("__half", 8, 1), ("__half", 32, 1), ("__half", 8, 2)]
# Most bytes of spill stores by chunks per lane: what four loads in flight beside one partial sum per
# chunk took at this bound (48 registers).  Eight loads beside two sums take 1,848 to 5,056.
LIMIT = {1: 660, 2: 1284}


def nvcc():
    try:
        return build.nvcc()
    except RuntimeError:
        return None


@pytest.mark.skipif(nvcc() is None, reason="no nvcc")
@pytest.mark.parametrize("storage,lanes,chunks", SHAPES)
def test_spill_stores(storage, lanes, chunks, tmp_path):
    src = tmp_path / "shape.cu"
    src.write_text('#include "sweep_kernels.cuh"\n'
                   f"template __global__ void ad::k_sweep<{storage}, {lanes}, {chunks}, false>(ad::SweepArgs);\n")
    r = subprocess.run([nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-I", build.CSRC, "-Xptxas", "-v", "-c", str(src),
                        "-o", os.devnull], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    found = re.search(r"Function properties for \S*k_sweep\S*\s+.*?(\d+) bytes spill stores", r.stderr)
    assert found, r.stderr
    assert int(found[1]) <= LIMIT[chunks]
