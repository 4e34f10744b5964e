"""The fine SGM's forms on the GPU: the default choice of scanlines to split across a CTA against no split
(the same bits), and two scanlines a warp (images with few wide windows) against the oracle."""
import numpy as np
import pytest

import lfsynth
import oracle
from lf_helpers import RTOL, csr_rel_err, gather, grad_tol, pad4_offsets
from test_gpu_backward import _cs_max, _elem_errors, _penalties, _run_gpu_backward
from test_gpu_parity import _dev, _gpu_sgm, _np

pytestmark = pytest.mark.gpu


def _windows(H, W, G, seed, wide_rows, wide_cols):
    """Random narrow windows, the given rows and columns of the whole range, and the CSR offsets."""
    rng = np.random.default_rng(seed)
    lo = rng.integers(0, G, (H, W)).astype(np.int32)
    cnt = np.minimum(rng.integers(1, 33, (H, W)), G - lo).astype(np.int32)
    for sel in [np.s_[r, :] for r in wide_rows] + [np.s_[:, c] for c in wide_cols]:
        lo[sel], cnt[sel] = 0, G
    lo, cnt = lo.ravel(), cnt.ravel()
    off = pad4_offsets(cnt)
    cost = np.zeros(int(off[-1]), np.float32)
    cost[np.repeat(off[:-1], cnt) + (np.arange(int(cnt.sum())) - np.repeat(np.cumsum(cnt) - cnt, cnt))] = \
        rng.uniform(0, 30, int(cnt.sum())).astype(np.float32)
    return lo, cnt, off, cost


# a direction of 256 pixels (the default splits from 24 wide windows on) and of 255 (it splits nothing);
# 23 wide windows on most of a row's scanlines, whole rows and columns, and more than 256 listed scanlines
@pytest.mark.parametrize("H,W,rows,cols", [(20, 256, [0, 7], [3]), (256, 17, [30], [16]), (20, 255, [0], []),
                                           (40, 256, [], list(range(20, 43))), (300, 260, range(0, 280), [])])
@pytest.mark.parametrize("penalties", [(-1.0, -1.0), (1.5, 9.0)])
def test_default_split_gives_the_same_bits_as_none(gpu_lib, H, W, rows, cols, penalties):
    import torch
    G = 75
    lo, cnt, off, cost = _windows(H, W, G, H + W, rows, cols)
    p = lfsynth.LFParams(U=3, V=3, H=H, W=W, census_w=5, dmin=-2.0, dmax=2.0, coarse_labels=32, fine_labels=G,
                         fine_radius=5)
    d = [_dev(cost), _dev(lo, torch.int32), _dev(cnt, torch.int32), _dev(off)]
    h = gpu_lib.lfsgm_create(p)
    out = []
    for min_wide in (0, 1 << 30, 0):
        gpu_lib.lfsgm_set_sgm_split(h, min_wide)
        agg = torch.full_like(d[0], float("nan"))
        gpu_lib.lfsgm_sgm_aggregate(h, *d, *penalties, agg)
        out.append(agg)
    gpu_lib.lfsgm_sync(h)
    gpu_lib.lfsgm_destroy(h)
    pad = np.ones(cost.size, bool)
    pad[np.repeat(off[:-1], cnt) + (np.arange(int(cnt.sum())) - np.repeat(np.cumsum(cnt) - cnt, cnt))] = False
    assert np.all(np.isfinite(_np(out[0])[~pad])) and np.all(_np(out[0])[pad] == 0.0)
    assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])


def _case(H, W, paths, kind, G=97):
    """Windows that stand still or step by a label, or that jump, of 1 to 32 labels; 'jumps' and 'rows' with
    wider ones (0.6 % of the pixels; two whole rows)."""
    p = lfsynth.LFParams(U=3, V=3, H=H, W=W, census_w=5, dmin=-2.0, dmax=2.0, coarse_labels=9, fine_labels=G,
                         fine_radius=8, w_l2=1.0, w_census=1.0 / 24, subpixel=2, softmin_tau=0.1, paths=paths)
    rng = np.random.default_rng(H * W + paths)
    if kind == "still":                            # one row's window length, drifting by a label now and then
        cnt = np.repeat(rng.integers(15, 33, H), W)
        lo = np.clip(20 + np.cumsum(rng.choice([-1, 0, 0, 0, 1], size=(H, W)), axis=1), 0, G - 33).ravel()
    else:
        cnt = rng.choice(np.array([1, 5, 31, 32, 33, 70]), size=H * W,
                         p=[.1, .2, .35, .344, .003, .003] if kind == "jumps" else [.1, .2, .35, .35, 0, 0])
        lo = (rng.random(H * W) * (G - cnt + 1)).astype(int)
        if kind == "rows":
            lo.reshape(H, W)[[0, H // 2]], cnt.reshape(H, W)[[0, H // 2]] = 0, G
    views = rng.uniform(0.0, 1.0, (p.V, p.U, H, W)).astype(np.float32)
    return p, views, lo.astype(np.int32), cnt.astype(np.int32), rng.normal(size=H * W).astype(np.float32)


# an even and an odd number of scanlines; scanlines of unequal length share a warp at the corners; 1 x 1100:
# scanlines of one pixel
@pytest.mark.parametrize("H,W,paths", [(20, 260, 16), (37, 257, 8), (330, 361, 8), (1, 1100, 8)])
@pytest.mark.parametrize("kind", ["still", "jumps"])
def test_two_scanlines_a_warp_match_the_oracle(gpu_lib, H, W, paths, kind):
    p, _, lo, cnt, _ = _case(H, W, paths, kind)
    assert np.sum(cnt > 32) <= H * W // 100
    off_o = oracle.offsets(cnt)
    cost = np.random.default_rng(3).uniform(0, 30, int(off_o[-1])).astype(np.float32)
    P1, P2 = np.float32(1.7), np.float32(9.5)
    Cs = oracle.sgm_bounded(H, W, lo, cnt, off_o, cost.astype(np.float64), float(P1), float(P2), paths)
    off, agg = _gpu_sgm(gpu_lib, p, cost, lo, cnt, P1, P2)
    err = csr_rel_err(gather(agg, off, cnt), Cs, cnt)
    assert err < RTOL, err


# The branches that split scanlines record, and the adjoint's wide steps (four labels a lane, 512 a round;
# 97, 98, 100 and 601 labels): the adjoint against the oracle's.  The bar is that of the other
# adjoint tests, for all but 1e-4 of the elements (decisions that FP32 rounding makes at a kink, as on the
# bench band).
@pytest.mark.parametrize("H,W,G", [(20, 260, 97), (260, 21, 98), (12, 60, 100), (6, 40, 601)])
def test_split_scanlines_record_the_adjoints_branches(gpu_lib, H, W, G):
    p, views, lo, cnt, gd = _case(H, W, 8, "rows", G)
    cfg = oracle.make_cfg(p)
    off_o, cost_o = oracle.cost_volume(cfg, views, lo, cnt)
    P1, P2 = _penalties(cost_o)
    gC_o, g1_o, g2_o, gV_o = oracle.backward(cfg, views, lo, cnt, cost_o, float(P1), float(P2), gd, p.softmin_tau)
    gC, g1, g2, gV = _run_gpu_backward(gpu_lib, p, views, lo, cnt, P1, P2, gd, p.softmin_tau, True)
    eC, eV = _elem_errors(p, cnt, gC, gC_o, gV, gV_o)
    tol = grad_tol(_cs_max(p, lo, cnt, off_o, cost_o, P1, P2), p.softmin_tau)
    assert np.mean(eC > tol) <= 1e-4 and np.mean(eV > tol) <= 1e-4
    assert np.abs(gC - gC_o).sum() <= 1e-3 * np.abs(gC_o).sum()


# the threshold: the library's own on a new handle (24 from 256 pixels in a direction on, not for whole-range searches),
# 0 for none, the caller's or the autotuner's; lfsgm_get_sgm_split reads back what was set
@pytest.mark.parametrize("H,W,boundless,own", [(20, 256, 0, 24), (256, 20, 0, 24), (255, 255, 0, 0), (20, 300, 1, 0)])
def test_split_threshold_in_use(gpu_lib, H, W, boundless, own):
    import torch
    p = lfsynth.LFParams(U=3, V=3, H=H, W=W, census_w=5, dmin=-2.0, dmax=2.0, coarse_labels=40, fine_labels=75,
                         fine_radius=5, boundless=boundless)
    h = gpu_lib.lfsgm_create(p)
    assert gpu_lib.lfsgm_get_sgm_split(h) == 0 and gpu_lib.lfsgm_sgm_split_used(h) == own
    for n in (0, 24, 7, 0):
        gpu_lib.lfsgm_set_sgm_split(h, n)
        assert gpu_lib.lfsgm_get_sgm_split(h) == n and gpu_lib.lfsgm_sgm_split_used(h) == n
    gpu_lib.lfsgm_set_sgm_split(h, 5)
    gpu_lib.lfsgm_autotune(h, _dev(lfsynth.random_views(3, 3, H, W, seed=H)))
    assert gpu_lib.lfsgm_get_sgm_split(h) == gpu_lib.lfsgm_sgm_split_used(h) and gpu_lib.lfsgm_get_sgm_split(h) in (0, 24)
    gpu_lib.lfsgm_destroy(h)
    v = torch.from_numpy(lfsynth.random_views(3, 3, H, W, seed=H)).cuda()
    b = gpu_lib.LightFieldBatch([p, p], [v, v], branches=1)
    assert b.knobs()[3].tolist() == [own, own]
    b.close()


# a new handle (two scanlines a warp, split from 24 on) against no split, one scanline a warp
@pytest.mark.parametrize("H,W,rows,cols", [(20, 256, [0, 7], [3]), (256, 17, [30], [16]), (40, 256, [], list(range(20, 43))),
                                           (300, 260, [0], []), (300, 260, range(0, 280), [])])
@pytest.mark.parametrize("penalties", [(-1.0, -1.0), (1.5, 9.0)])
def test_new_handle_gives_the_bits_of_no_split(gpu_lib, H, W, rows, cols, penalties):
    import torch
    G = 75
    lo, cnt, off, cost = _windows(H, W, G, H + W, [r for r in rows if r < H], cols)
    p = lfsynth.LFParams(U=3, V=3, H=H, W=W, census_w=5, dmin=-2.0, dmax=2.0, coarse_labels=40, fine_labels=G,
                         fine_radius=5)
    d = [_dev(cost), _dev(lo, torch.int32), _dev(cnt, torch.int32), _dev(off)]
    h = gpu_lib.lfsgm_create(p)
    out = []
    for min_wide in (None, 0, 24, 1 << 30, 0):
        if min_wide is not None:
            gpu_lib.lfsgm_set_sgm_split(h, min_wide)
        agg = torch.full_like(d[0], float("nan"))
        gpu_lib.lfsgm_sgm_aggregate(h, *d, *penalties, agg)
        out.append(agg)
    gpu_lib.lfsgm_sync(h)
    gpu_lib.lfsgm_destroy(h)
    assert all(torch.equal(out[0], a) for a in out[1:])


# a share of wide windows at which scanlines run two to a warp in images of any shape (0.3 %), and more: both forms
@pytest.mark.parametrize("H,W,paths", [(20, 260, 16), (37, 257, 8), (330, 361, 8), (300, 310, 16)])
@pytest.mark.parametrize("share", [0.003, 0.02, 0.3])
def test_wide_windows_by_share_match_the_oracle(gpu_lib, H, W, paths, share):
    G = 97
    p, _, lo, cnt, _ = _case(H, W, paths, "narrow", G)
    rng = np.random.default_rng(int(share * 1000) + W)
    wide = rng.random(H * W) < share
    cnt[wide] = rng.integers(33, 90, int(wide.sum()))
    lo = np.minimum(lo, G - cnt).astype(np.int32)
    off_o = oracle.offsets(cnt)
    cost = np.random.default_rng(3).uniform(0, 30, int(off_o[-1])).astype(np.float32)
    P1, P2 = np.float32(1.7), np.float32(9.5)
    Cs = oracle.sgm_bounded(H, W, lo, cnt, off_o, cost.astype(np.float64), float(P1), float(P2), paths)
    for split in (None, 0):
        off, agg = _gpu_sgm(gpu_lib, p, cost, lo, cnt, P1, P2) if split == 0 else _new_handle_sgm(gpu_lib, p, cost, lo, cnt, P1, P2)
        err = csr_rel_err(gather(agg, off, cnt), Cs, cnt)
        assert err < RTOL, (split, err)


def _new_handle_sgm(gpu_lib, p, cost, lo, cnt, P1, P2):
    """As _gpu_sgm, on a handle whose split is not set."""
    import torch
    off = pad4_offsets(cnt)
    full = np.zeros(int(off[-1]), np.float32)
    full[np.repeat(off[:-1], cnt) + (np.arange(int(cnt.sum())) - np.repeat(np.cumsum(cnt) - cnt, cnt))] = cost
    cd = _dev(full)
    h = gpu_lib.lfsgm_create(p)
    agg = torch.full_like(cd, float("nan"))
    gpu_lib.lfsgm_sgm_aggregate(h, cd, _dev(lo, torch.int32), _dev(cnt, torch.int32), _dev(off), P1, P2, agg)
    gpu_lib.lfsgm_sync(h)
    gpu_lib.lfsgm_destroy(h)
    return off, _np(agg)


# 160 scanlines that cross 26 wide windows each: too many to split on a new handle, unless one crosses 96 (the whole row)
@pytest.mark.parametrize("long_row", [False, True])
@pytest.mark.parametrize("record", [False, True])
def test_many_listed_scanlines_give_the_bits_of_no_split(gpu_lib, long_row, record):
    import torch
    H, W, G = 300, 260, 75
    rng = np.random.default_rng(9)
    lo = rng.integers(0, G, (H, W)).astype(np.int32)
    cnt = np.minimum(rng.integers(1, 33, (H, W)), G - lo).astype(np.int32)
    for y in range(80):
        x = 3 * y % 230
        lo[y, x:x + 26], cnt[y, x:x + 26] = 0, G
    if long_row:
        lo[200], cnt[200] = 0, G
    lo, cnt = lo.ravel(), cnt.ravel()
    off = pad4_offsets(cnt)
    cost = rng.uniform(0, 30, int(off[-1])).astype(np.float32)
    p = lfsynth.LFParams(U=3, V=3, H=H, W=W, census_w=5, dmin=-2.0, dmax=2.0, coarse_labels=40, fine_labels=G,
                         fine_radius=5)
    d = [_dev(cost), _dev(lo, torch.int32), _dev(cnt, torch.int32), _dev(off)]
    h = gpu_lib.lfsgm_create(p)
    out = []
    for min_wide in (None, 0, 24):
        if min_wide is not None:
            gpu_lib.lfsgm_set_sgm_split(h, min_wide)
        agg = torch.full_like(d[0], float("nan"))
        (gpu_lib.lfsgm_sgm_aggregate_record if record else gpu_lib.lfsgm_sgm_aggregate)(h, *d, 1.5, 9.0, agg)
        out.append(agg)
    gpu_lib.lfsgm_sync(h)
    gpu_lib.lfsgm_destroy(h)
    assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])


@pytest.mark.parametrize("radius,far,own", [(15, 0, 24), (16, 0, 0), (5, 16, 0)])
def test_no_split_of_its_own_where_the_regular_windows_are_wide(gpu_lib, radius, far, own):
    p = lfsynth.LFParams(U=3, V=3, H=20, W=260, census_w=5, dmin=-2.0, dmax=2.0, coarse_labels=40, fine_labels=75,
                         fine_radius=radius, fine_radius_far=far)
    h = gpu_lib.lfsgm_create(p)
    assert gpu_lib.lfsgm_sgm_split_used(h) == own
    gpu_lib.lfsgm_destroy(h)
