"""The work counted for the emulated trailing update: the tiles that the kernel visits, the
right-hand side's row included, and the rate of the slice products that it executes."""
import os
import re
import sys

import pytest

from synth.configs import small

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
TILE = 8 * 36 * 2 * (2 * 16 * 8 * 16)


def _sizes(w):
    from paper_2103_08513_gb300 import MRCM
    return MRCM(w.n, w.edges, w.patch, precision="fp64", allocate=False).sizes


# one front of 2 x faces eliminated dofs, panels of 32: (m, tiles) of the steps with m >= 24
# 32: m = 32, rows 0 .. 32 (the last one right-hand side): tiles (0, 0), (1, 0)
# 33: m = 34: three; 48: m = 64 (5), m = 32 (2); 47: m = 62 (3), m = 30 (1)
@pytest.mark.parametrize("faces,tiles", [(32, 2), (33, 3), (48, 7), (47, 4)])
def test_tiles_of_one_front(faces, tiles):
    w = small(n=(6, faces, 2), edges=([3, 3], [faces], [2]), patch=((1, 2), (1, 1), (1, 1)))
    assert _sizes(w)["ldl_update_tensor_flops"] == tiles * TILE


def test_executed_rate_follows_the_kernels_slices():
    sys.path.insert(0, ROOT)
    import bench
    src = open(os.path.join(ROOT, "paper_2103_08513_gb300", "csrc", "mrcm_interface.cu")).read()
    S = int(re.search(r"constexpr int kOzS = (\d+);", src).group(1))
    assert bench.LDL_EXECUTED == S * (S + 1) / 2 / 36
    peaks = {"hbm_gbs": 6000.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0, "fp32_tflops": 80.0,
             "fp64_tflops": 1.0, "fp64_source": "test", "source": "test"}
    sizes = {"ldl_update_tensor_flops": 36e12, "n_cells": 1}
    r = bench.roofline("k_ldl_update", 1000.0, 1, 1, sizes, 0, "fp32_ir", peaks)
    assert r["achieved"] == 36.0 and abs(r["executed"] - 28.0) < 1e-9 and abs(r["executed_frac"] - 28.0 / 1700.0) < 1e-4
