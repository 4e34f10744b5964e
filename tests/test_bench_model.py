"""Host-side models of bench.py: the row cost kernel's choice of windows (replayed on the host to
count the cells it computes) on hand-made window maps."""
import numpy as np

import bench


def test_row_kernel_cells_hand_cases():
    H, W = 1, 64
    lo = np.zeros(W, np.int32)
    cnt = np.full(W, 31, np.int32)
    # first run of 32 pixels: all windows start at 10 except one at 50 (outside 10 .. 45) and one
    # wide window (40 labels): 30 windows of 31 labels fit
    lo[:32] = 10
    lo[5] = 50
    cnt[7] = 40
    # second run: starts 0..5 and 6 alternate; [0, 36) holds starts 0..5 with 31 labels
    lo[32:] = np.arange(32) % 7
    got = bench.row_kernel_cells(lo, cnt, H, W)
    second = int(sum(31 for i in range(32) if lo[32 + i] + 31 <= 36))
    assert got == 30 * 31 + second
    # a run without narrow windows contributes nothing
    assert bench.row_kernel_cells(np.zeros(32, np.int32), np.full(32, 40, np.int32), 1, 32) == 0


def test_row_kernel_cells_prefers_the_lowest_start_on_ties():
    # two groups of 16 windows (starts 0 and 40, 31 labels): equal fits, the lower start wins
    lo = np.where(np.arange(32) < 16, 40, 0).astype(np.int32)
    cnt = np.full(32, 31, np.int32)
    cnt[0] = 20                                     # a narrower window in the start-40 group
    got = bench.row_kernel_cells(lo, cnt, 1, 32)
    assert got == 16 * 31


def test_dominant_kernel_is_among_the_kernels_the_stages_launch():
    import os
    import re
    api = open(os.path.join(os.path.dirname(bench.__file__), "paper_1907_13449_gb300", "csrc", "lfsgm_api.cu")).read()

    def launched(start, end):
        return set(re.findall(r'run\(h, "(\w+)"', api[api.index(start):api.index(end)]))
    stages = launched("lfsgm_status cost_volume_impl(", "\nint *split_table") | launched("lfsgm_status lfsgm_sgm_aggregate(", "lfsgm_status lfsgm_wta_subpixel(")
    assert set(bench.COST_SGM_KERNELS) == stages - {"set_penalties"}    # (explicit penalties only)
    ms = dict(census_all=0.03, fine_cost=0.01, fine_cost_runs=0.17, fine_cost_census=0.02, fine_cost_wide=0.2, fine_sgm=0.1,
              coarse_sgm=0.5)
    kernels = {k: {"ms_total": v} for k, v in ms.items()}
    assert bench.dominant_kernel(kernels) == "fine_cost_runs"
    del kernels["fine_cost_census"]
    assert bench.dominant_kernel(kernels) == "fine_cost_wide"
