"""The row cost kernel (k_fine_rows.cu): its square root against sqrtf, and its blocks, tasks and list
at sizes where they can go wrong, against the FP64 oracle."""
import os
import subprocess

import numpy as np
import pytest

import lfsynth
import oracle
from lf_helpers import RTOL, csr_rel_err, gather, pad4_offsets

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_sqrt_fast_rounds_as_sqrtf(tmp_path):
    from paper_1907_13449_gb300 import _build
    exe = str(tmp_path / "sqrt_check")
    subprocess.run([_build.nvcc(), "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "-I", _build.CSRC,
                    "-o", exe, os.path.join(HERE, "sqrt_check.cu")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "0", (r.returncode, r.stdout, r.stderr)


# image sizes around the 32 x 8 blocks; windows: nearly equal rows (one task a block), rows that differ
# by more than a task's span (several tasks, and rows left to the list), and single odd windows
@pytest.mark.parametrize("channels", [1, 3])
@pytest.mark.parametrize("H,W", [(1, 1), (7, 33), (8, 32), (9, 31), (17, 65)])
@pytest.mark.parametrize("kind", ["even", "rows", "mixed"])
def test_blocks_and_tasks_match_the_oracle(gpu_lib, H, W, kind, channels):
    import torch
    G = 121
    p = lfsynth.LFParams(U=3, V=4, H=H, W=W, census_w=5, dmin=-3.0, dmax=3.0, coarse_labels=16, fine_labels=G,
                         fine_radius=7, channels=channels)
    rng = np.random.default_rng(H * 1000 + W + channels)
    views = lfsynth.random_views(p.U, p.V, H, W, seed=H + W, channels=channels)
    y, x = np.mgrid[0:H, 0:W]
    if kind == "even":
        lo = 40 + (x + y) % 3
        cnt = np.full((H, W), 31)
    elif kind == "rows":
        lo = (y % 8) * 13 + rng.integers(0, 3, (H, W))       # starts 0 .. 93: eight spans in a block
        cnt = rng.integers(5, 28, (H, W))
    else:
        lo = rng.integers(0, G, (H, W))
        cnt = rng.integers(1, G + 1, (H, W))
        cnt = np.where(rng.random((H, W)) < 0.7, np.minimum(cnt, 32), cnt)
    lo = lo.astype(np.int32).reshape(-1)
    cnt = np.minimum(cnt.reshape(-1), G - lo).astype(np.int32)
    off = pad4_offsets(cnt)
    L = gpu_lib.LightFieldDepth(p)
    L.lo.copy_(torch.from_numpy(lo))
    L.cnt.copy_(torch.from_numpy(cnt))
    L.off.copy_(torch.from_numpy(off))
    L.cost.fill_(float("nan"))
    L.cost_volume(torch.from_numpy(views).cuda())
    gpu_lib.lfsgm_sync(L.h)
    got = L.cost.cpu().numpy()
    L.close()
    off_o, ref = oracle.cost_volume(oracle.make_cfg(p), views, lo, cnt)
    assert csr_rel_err(gather(got, off, cnt), gather(ref, off_o, cnt), cnt) <= RTOL
    pad = np.ones(off[-1], bool)
    pad[np.repeat(off[:-1], cnt) + np.arange(cnt.sum()) - np.repeat(np.cumsum(cnt) - cnt, cnt)] = False
    assert not np.any(got[:off[-1]][pad])                    # padding slots are 0


def _rgb_costs(gpu_lib, p, views, lo, cnt):
    """The colour cost volume's active slots in the row kernel and, with span 44, in the list kernel."""
    import torch
    off = pad4_offsets(cnt)
    out = []
    for kw in (36, 44):
        L = gpu_lib.LightFieldDepth(p)
        gpu_lib.lfsgm_set_tuning(L.h, kw)
        L.lo.copy_(torch.from_numpy(lo))
        L.cnt.copy_(torch.from_numpy(cnt))
        L.off.copy_(torch.from_numpy(off))
        L.cost_volume(torch.from_numpy(views).cuda())
        gpu_lib.lfsgm_sync(L.h)
        out.append(gather(L.cost.cpu().numpy(), off, cnt))
        L.close()
    return out


def _rgb_case(**kw):
    p = lfsynth.LFParams(U=3, V=4, H=9, W=37, census_w=5, dmin=-3.0, dmax=3.0, coarse_labels=16, fine_labels=121,
                         fine_radius=7, channels=3, **kw)
    y, x = np.mgrid[0:p.H, 0:p.W]
    lo = (40 + (x + y) % 3).astype(np.int32).reshape(-1)
    return p, lfsynth.random_views(p.U, p.V, p.H, p.W, seed=4, channels=3), lo, np.full(p.N, 31, np.int32)


def test_colour_costs_of_huge_differences_are_infinite_not_nan(gpu_lib):
    """A reference value whose squared difference overflows gives +inf (also an infinite one), a NaN NaN, and
    1e19, whose squares' sum does not overflow, its norm; in both kernels.  The other pixels do not change."""
    p, views, lo, cnt = _rgb_case(w_census=0.0)
    _, ref = oracle.cost_volume(oracle.make_cfg(p), views, lo, cnt)
    ref = ref.reshape(p.N, 31)
    bad = {3: 1e25, 40: -1e25, 77: np.inf, 130: -np.inf, 200: np.nan, 290: 1e19}
    for q, v in bad.items():
        views[p.vc, p.uc, :1 if q == 40 else 3].reshape(-1, p.N)[:, q] = v
    for got in _rgb_costs(gpu_lib, p, views, lo, cnt):
        got = got.reshape(p.N, 31)
        for q, v in bad.items():
            if np.isnan(v):
                assert np.all(np.isnan(got[q]))
            elif abs(v) > 1e20:
                assert np.all(np.isposinf(got[q])), (q, v, got[q])
            else:
                assert np.allclose(got[q], (p.U * p.V - 1) * np.sqrt(3.0) * v, rtol=RTOL, atol=0.0)
        same = np.setdiff1d(np.arange(p.N), list(bad))
        assert csr_rel_err(got[same].ravel(), ref[same].ravel(), cnt[same]) <= RTOL


# FP32 scales exactly by powers of two until a squared norm has less than 24 bits left: at 2^-63 a difference of
# 0.01 or more of the range loses at most 2^-12 of itself, below 1e-6 of its pixel's sum
@pytest.mark.parametrize("scale", [2.0 ** -20, 2.0 ** -50, 2.0 ** -63, 2.0 ** 50])
def test_colour_costs_scale_with_the_views(gpu_lib, scale):
    p, views, lo, cnt = _rgb_case(w_census=0.0)
    views = (views * np.float32(scale)).astype(np.float32)
    _, ref = oracle.cost_volume(oracle.make_cfg(p), views, lo, cnt)
    for got in _rgb_costs(gpu_lib, p, views, lo, cnt):
        assert csr_rel_err(got, ref, cnt) <= RTOL


# more tasks than CTAs: rows of eight different spans in each of 175 blocks (1400 tasks, 783 CTAs), so that a CTA
# runs a second task on barriers set up anew, with rows that have no pixel in it
@pytest.mark.parametrize("channels", [1, 3])
def test_more_tasks_than_ctas_match_the_oracle(gpu_lib, channels):
    import torch
    H = W = 200
    p = lfsynth.LFParams(U=3, V=4, H=H, W=W, census_w=5, dmin=-3.0, dmax=3.0, coarse_labels=16, fine_labels=441,
                         fine_radius=7, channels=channels)
    rng = np.random.default_rng(7 + channels)
    views = lfsynth.random_views(p.U, p.V, H, W, seed=11, channels=channels)
    y = np.repeat(np.arange(H), W)
    lo = ((y % 8) * 52 + rng.integers(0, 3, H * W)).astype(np.int32)    # starts at least 50 apart: a task a row
    cnt = rng.integers(5, 29, H * W).astype(np.int32)
    off = pad4_offsets(cnt)
    L = gpu_lib.LightFieldDepth(p)
    L.lo.copy_(torch.from_numpy(lo))
    L.cnt.copy_(torch.from_numpy(cnt))
    L.off.copy_(torch.from_numpy(off))
    off_o, ref = oracle.cost_volume(oracle.make_cfg(p), views, lo, cnt)
    for _ in range(2):
        L.cost.fill_(float("nan"))
        L.cost_volume(torch.from_numpy(views).cuda())
        gpu_lib.lfsgm_sync(L.h)
        assert csr_rel_err(gather(L.cost.cpu().numpy(), off, cnt), gather(ref, off_o, cnt), cnt) <= RTOL
    L.close()


def test_ranges_whose_boxes_just_fit_take_the_row_kernel(gpu_lib):
    """A range of 36 labels over 200 pixels (a row of nine views): 40 labels would not fit a 256-wide box, so tasks
    span the 36 labels of a row's own range."""
    import torch
    G = 81
    p = lfsynth.LFParams(U=9, V=1, H=19, W=97, census_w=5, dmin=-57.0, dmax=57.0, coarse_labels=16, fine_labels=G,
                         fine_radius=7)
    rng = np.random.default_rng(3)
    views = lfsynth.random_views(p.U, p.V, p.H, p.W, seed=2)
    lo = rng.integers(0, G, p.N).astype(np.int32)
    lo[:p.N // 2] = 20 + lo[:p.N // 2] % 5
    cnt = np.minimum(rng.integers(5, 33, p.N), G - lo).astype(np.int32)
    off = pad4_offsets(cnt)
    L = gpu_lib.LightFieldDepth(p)
    L.lo.copy_(torch.from_numpy(lo))
    L.cnt.copy_(torch.from_numpy(cnt))
    L.off.copy_(torch.from_numpy(off))
    vd = torch.from_numpy(views).cuda()
    gpu_lib.lfsgm_set_profiling(L.h, True)
    L.cost_volume(vd)
    gpu_lib.lfsgm_sync(L.h)
    assert "row_tasks" in [n for n, _ in gpu_lib.lfsgm_kernel_times(L.h)]
    got = L.cost.cpu().numpy()
    L.close()
    off_o, ref = oracle.cost_volume(oracle.make_cfg(p), views, lo, cnt)
    assert csr_rel_err(gather(got, off, cnt), gather(ref, off_o, cnt), cnt) <= RTOL


# images of more than 152 blocks, whose tasks are of up to eight rows (fewer in smaller ones), with ragged edges
@pytest.mark.parametrize("channels", [1, 3])
@pytest.mark.parametrize("kind", ["even", "mixed"])
def test_tasks_of_eight_rows_match_the_oracle(gpu_lib, kind, channels):
    import torch
    H, W, G = 203, 205, 121
    p = lfsynth.LFParams(U=3, V=4, H=H, W=W, census_w=5, dmin=-3.0, dmax=3.0, coarse_labels=16, fine_labels=G,
                         fine_radius=7, channels=channels)
    rng = np.random.default_rng(20 + channels)
    views = lfsynth.random_views(p.U, p.V, H, W, seed=21, channels=channels)
    y, x = np.mgrid[0:H, 0:W]
    lo = (40 + (x + y) % 3).ravel() if kind == "even" else rng.integers(0, G, H * W)
    cnt = np.full(H * W, 31) if kind == "even" else np.where(rng.random(H * W) < 0.1, G, rng.integers(1, 33, H * W))
    lo = lo.astype(np.int32)
    cnt = np.minimum(cnt, G - lo).astype(np.int32)
    off = pad4_offsets(cnt)
    L = gpu_lib.LightFieldDepth(p)
    L.lo.copy_(torch.from_numpy(lo))
    L.cnt.copy_(torch.from_numpy(cnt))
    L.off.copy_(torch.from_numpy(off))
    L.cost_volume(torch.from_numpy(views).cuda())
    gpu_lib.lfsgm_sync(L.h)
    got = L.cost.cpu().numpy()
    L.close()
    off_o, ref = oracle.cost_volume(oracle.make_cfg(p), views, lo, cnt)
    assert csr_rel_err(gather(got, off, cnt), gather(ref, off_o, cnt), cnt) <= RTOL
