"""The end of the initial pass on the GPU: fusion, filling and windows in one kernel (up to two filling
passes, 32 x 8 tiles with a halo) or in several, and the offsets' scan, each exactly as the oracle's."""
import numpy as np
import pytest

import lfsynth
import oracle
from lf_helpers import pad4_offsets
from test_gpu_parity import _check_initial, _dev, _np

pytestmark = pytest.mark.gpu


# one pixel row beyond a tile, exactly a tile, one column beyond, several tiles; phi = 0.5 leaves holes of
# many pixels, so that values from the whole halo reach a pixel
@pytest.mark.parametrize("H,W", [(9, 32), (8, 32), (17, 33), (40, 101)])
@pytest.mark.parametrize("passes", [0, 1, 2, 3])
def test_windows_after_filling_match_the_oracle(gpu_lib, H, W, passes):
    import torch
    p = lfsynth.tiny_params(U=3, V=3, H=H, W=W, coarse_labels=40, fill_passes=passes, phi=0.5,
                            edge_threshold=1.5 if passes == 2 else 0.0)
    views, _, p = lfsynth.tiny(params=p)
    other, _, _ = lfsynth.tiny(1, params=p)
    N = p.H * p.W
    lo = torch.empty(N, dtype=torch.int32, device="cuda")
    cnt = torch.empty_like(lo)
    off = torch.empty(N + 1, dtype=torch.int64, device="cuda")
    dinit = torch.empty(N, dtype=torch.float32, device="cuda")
    maps = torch.full((4, N), -7, dtype=torch.int32, device="cuda")
    h = gpu_lib.lfsgm_create(p)
    for v in (other, views):                           # the second call finds the first one's sums
        nnz = gpu_lib.lfsgm_initial_disparity(h, _dev(v), 0, 0, lo, cnt, off, dinit, maps, want_nnz=True)
    gpu_lib.lfsgm_sync(h)
    gpu_lib.lfsgm_destroy(h)
    ref = oracle.initial_disparity(oracle.make_cfg(p), views, None, p.p1_frac, p.p2_frac)
    _check_initial(dict(lo=_np(lo), cnt=_np(cnt), off=_np(off), dinit=_np(dinit), maps=_np(maps), nnz=nnz), ref, p)


# one scan tile and a pixel more, and more tiles than one CTA adds up (1024 of 1024 pixels)
@pytest.mark.parametrize("H,W", [(41, 25), (1027, 1024)])
def test_offsets_are_the_padded_counts_prefix_sums(gpu_lib, H, W):
    import torch
    p = lfsynth.tiny_params(U=3, V=1, H=H, W=W, coarse_labels=8, fine_labels=21)
    views = np.random.default_rng(H).random((p.V, p.U, H, W)).astype(np.float32)
    N = H * W
    lo = torch.empty(N, dtype=torch.int32, device="cuda")
    cnt = torch.empty_like(lo)
    off = torch.empty(N + 1, dtype=torch.int64, device="cuda")
    h = gpu_lib.lfsgm_create(p)
    gpu_lib.lfsgm_initial_disparity(h, _dev(views), 0, 0, lo, cnt, off, None, None)
    gpu_lib.lfsgm_sync(h)
    gpu_lib.lfsgm_destroy(h)
    assert len(np.unique(_np(cnt))) > 1
    assert np.array_equal(_np(off), pad4_offsets(_np(cnt)))


# taller than 65535 tiles of eight rows: the windows of a column of views and of its transpose, a row
def test_windows_of_a_very_tall_image_are_its_transposes(gpu_lib):
    import torch
    N = 8 * 65535 + 9
    views = np.random.default_rng(5).random((2, N)).astype(np.float32)
    got = []
    for U, V, H, W in ((1, 2, N, 1), (2, 1, 1, N)):
        p = lfsynth.tiny_params(U=U, V=V, H=H, W=W, coarse_labels=33, fine_labels=21, fill_passes=2, phi=1.0)
        lo = torch.empty(N, dtype=torch.int32, device="cuda")
        cnt = torch.empty_like(lo)
        off = torch.empty(N + 1, dtype=torch.int64, device="cuda")
        h = gpu_lib.lfsgm_create(p)
        gpu_lib.lfsgm_initial_disparity(h, _dev(views.reshape(V, U, H, W)), 0, 0, lo, cnt, off, None, None)
        gpu_lib.lfsgm_sync(h)
        gpu_lib.lfsgm_destroy(h)
        got.append((_np(lo), _np(cnt), _np(off)))
    assert len(np.unique(got[0][0])) > 1 and np.array_equal(got[0][2], pad4_offsets(got[0][1]))
    for a, b in zip(*got):
        assert np.array_equal(a, b)
