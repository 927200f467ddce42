"""The committed ncu summary of the 2D batches' row sweep belongs to the current
source of that kernel (bench.py reports its DRAM traffic only then)."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


def test_committed_row_sweep_profile_matches_current_kernel():
    traffic = bench._traffic(bench._kernel_sha(2, "wlb_batch_2d.cu"), name="batch_rows_2d_d2q5_f32_ensemble512.md")
    assert traffic is not None, "kernel source changed since its profile was captured"
    # 40 B x 512 x 192^2 cells per launch of six steps; c^2 near the object on top,
    # some writes still dirty in L2 at the kernel's end
    assert 0.9 * 7.5497e8 < traffic < 1.1 * 7.5497e8
