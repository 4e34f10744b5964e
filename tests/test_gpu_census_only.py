"""The cost volume without the l2 term (w_l2 = 0): runs of whole-range windows, other windows and
views with non-finite values, against the oracle (integer Hamming sums, exact)."""
import numpy as np
import pytest

import lfsynth
import oracle
from lf_helpers import gather, pad4_offsets

pytestmark = pytest.mark.gpu


def _cost(lf, p, views, lo, cnt, off):
    import torch
    L = lf.LightFieldDepth(p)
    for t, a in ((L.lo, lo), (L.cnt, cnt), (L.off, off)):
        t.copy_(torch.from_numpy(a))
    L.cost.fill_(-1.0)
    L.cost_volume(torch.from_numpy(views).cuda())
    lf.lfsgm_sync(L.h)
    out = L.cost.cpu().numpy()[:off[-1]]
    L.close()
    return out


# label counts around the chunks of 96 and 32, rows around the runs of 32 pixels
@pytest.mark.parametrize("G", [33, 95, 96, 97, 121, 200])
@pytest.mark.parametrize("H,W", [(1, 1), (3, 32), (9, 33), (2, 70)])
@pytest.mark.parametrize("kind", ["whole", "mixed"])
def test_census_only_cost_matches_the_oracle(gpu_lib, G, H, W, kind):
    p = lfsynth.LFParams(U=5, V=2, H=H, W=W, census_w=7, dmin=0.0, dmax=7.0, coarse_labels=16, fine_labels=G,
                         fine_radius=5, boundless=1, w_l2=0.0, w_census=1.0)
    views = lfsynth.random_views(p.U, p.V, H, W, seed=G + W)
    rng = np.random.default_rng(G)
    lo, cnt = np.zeros(p.N, np.int32), np.full(p.N, G, np.int32)
    if kind == "mixed":
        odd = rng.random(p.N) < 0.05                     # most runs keep one other window, a few none
        lo[odd] = rng.integers(0, G - 1, odd.sum())
        cnt[odd] = np.minimum(rng.integers(1, G + 1, odd.sum()), G - lo[odd])
    off = pad4_offsets(cnt)
    got = _cost(gpu_lib, p, views, lo, cnt, off)
    off_o, ref = oracle.cost_volume(oracle.make_cfg(p), views, lo, cnt)
    assert np.array_equal(gather(got, off, cnt).astype(np.float64), gather(ref, off_o, cnt))
    rest = np.ones(off[-1], bool)
    rest[np.repeat(off[:-1], cnt) + np.arange(cnt.sum()) - np.repeat(np.cumsum(cnt) - cnt, cnt)] = False
    assert not np.any(got[rest])


def test_non_finite_views_keep_the_full_form(gpu_lib):
    """0 x l2 is NaN where a sample is infinite: such views run the full form."""
    p = lfsynth.LFParams(U=3, V=1, H=8, W=40, census_w=5, dmin=0.0, dmax=2.0, coarse_labels=8, fine_labels=41,
                         fine_radius=5, boundless=1, w_l2=0.0, w_census=1.0)
    views = lfsynth.random_views(p.U, p.V, p.H, p.W, seed=5)
    cnt = np.full(p.N, 41, np.int32)
    off = pad4_offsets(cnt)
    lo = np.zeros(p.N, np.int32)
    plain = _cost(gpu_lib, p, views, lo, cnt, off)
    assert np.isfinite(plain).all()
    views[0, 2, 4, 20] = np.inf
    got = _cost(gpu_lib, p, views, lo, cnt, off)
    bad = np.isnan(got)
    assert bad.any() and not bad.all()


def test_no_launch_for_runs_that_cannot_be(gpu_lib):
    """Up to 32 fine labels no window is wider than 32, so no run is marked: its kernel is left out; the costs are
    those of the oracle."""
    import torch
    p = lfsynth.LFParams(U=4, V=3, H=21, W=70, census_w=5, dmin=-2.0, dmax=2.0, coarse_labels=40, fine_labels=32,
                         fine_radius=3, w_l2=0.0, w_census=1.0, boundless=1)
    views = lfsynth.random_views(4, 3, p.H, p.W, seed=8)
    L = gpu_lib.LightFieldDepth(p)
    vd = torch.from_numpy(views).cuda()
    L.initial(vd)
    gpu_lib.lfsgm_set_profiling(L.h, True)
    L.cost_volume(vd)
    gpu_lib.lfsgm_sync(L.h)
    assert "fine_cost_runs" not in [n for n, _ in gpu_lib.lfsgm_kernel_times(L.h)]
    got = L.cost.cpu().numpy()[:p.N * 32].reshape(p.N, 32)
    L.close()
    lo, cnt = np.zeros(p.N, np.int32), np.full(p.N, 32, np.int32)
    _, ref = oracle.cost_volume(oracle.make_cfg(p), views, lo, cnt)
    assert np.array_equal(got.astype(np.float64).ravel(), ref)
