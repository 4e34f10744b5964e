"""The coarse SGM's forms (labels per lane, scanlines per warp, byte and 16-bit costs) at their edges:
the per-arm maps and the search windows against the oracle, integer for integer."""
import numpy as np
import pytest

import lfsynth
import oracle

pytestmark = pytest.mark.gpu


# label counts around the forms' limits (32, 64, 128 labels; full and part-filled groups of lanes), scanline
# counts that leave a warp's second group empty, rows shorter and longer than the copies in flight; 13 x 1
# and 13 x 13 views: arm costs above 255 (16-bit rows)
@pytest.mark.parametrize("Lc", [2, 31, 32, 33, 60, 61, 64, 65, 100, 124, 125, 128, 129, 248, 256])
@pytest.mark.parametrize("U,V,H,W,paths", [(3, 3, 5, 7, 8), (4, 1, 1, 40, 8), (3, 5, 29, 17, 16), (13, 1, 9, 33, 8)])
def test_coarse_maps_match_the_oracle(gpu_lib, Lc, U, V, H, W, paths):
    import torch
    p = lfsynth.LFParams(U=U, V=V, H=H, W=W, census_w=7, dmin=-1.5, dmax=1.5, coarse_labels=Lc, fine_labels=31,
                         fine_radius=4, paths=paths)
    views = lfsynth.random_views(U, V, H, W, seed=Lc + W)
    ref = oracle.initial_disparity(oracle.make_cfg(p), views, p1f=p.p1_frac, p2f=p.p2_frac)
    L = gpu_lib.LightFieldDepth(p)
    L.initial(torch.from_numpy(views).cuda())
    gpu_lib.lfsgm_sync(L.h)
    n = len(ref["arms"])
    assert np.array_equal(L.maps.cpu().numpy()[:n], np.asarray(ref["maps"]).reshape(n, -1))
    assert np.array_equal(L.lo.cpu().numpy(), ref["lo"]) and np.array_equal(L.cnt.cpu().numpy(), ref["cnt"])
    L.close()


# byte rows of two labels a lane (up to 32 labels), whose copies even lanes make for their odd neighbours: scanlines
# of many times the rows in flight, odd label counts, the same maps every time
@pytest.mark.parametrize("Lc", [3, 17, 30, 32])
@pytest.mark.parametrize("H,W,paths", [(33, 301, 8), (257, 19, 16)])
def test_copied_byte_rows_match_the_oracle_each_time(gpu_lib, Lc, H, W, paths):
    import torch
    p = lfsynth.LFParams(U=3, V=3, H=H, W=W, census_w=5, dmin=-1.5, dmax=1.5, coarse_labels=Lc, fine_labels=31,
                         fine_radius=4, paths=paths)
    views = lfsynth.random_views(3, 3, H, W, seed=Lc + W)
    ref = oracle.initial_disparity(oracle.make_cfg(p), views, p1f=p.p1_frac, p2f=p.p2_frac)
    L = gpu_lib.LightFieldDepth(p)
    n = len(ref["arms"])
    for _ in range(4):
        L.maps.fill_(-1)
        L.initial(torch.from_numpy(views).cuda())
        gpu_lib.lfsgm_sync(L.h)
        assert np.array_equal(L.maps.cpu().numpy()[:n], np.asarray(ref["maps"]).reshape(n, -1))
    L.close()
