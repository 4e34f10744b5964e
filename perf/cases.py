"""What is timed: the depth method and its stages on light fields of the sizes that it is used on.

A case is one call, or the few calls of one stage, on one light field (``batch``: on several), made
through the package's public functions.  ``kind`` says which:

  depth    the whole method on device views (lfsgm_depth)
  host     the whole method from pinned host views to a host disparity map (lfsgm_depth_host)
  initial  the initial pass: per-arm census matching and the search windows
  cost     the bounded cost volume on the windows of the initial pass
  sgm      the bounded SGM over a cost volume, with the penalties from its mean
  final    cost volume + SGM + winner / sub-pixel (the final map) on given windows
  train    a training step with the C-level calls: cost volume, recorded SGM, soft-argmin, backward
  autograd a training step through torch autograd, with learnable penalties
  batch    several light fields of mixed shape as one graph launch

The scenes are slanted textured planes on Voronoi cells with noise, rendered here on the GPU.
``exact`` computes a case's outputs in 64 bits with plain torch.
"""
import math

import torch

import paper_1907_13449_gb300 as lf

DEFAULTS = dict(U=9, V=9, H=512, W=512, census_w=7, dmin=-4.0, dmax=4.0, coarse_labels=100, fine_labels=401,
                fine_radius=15, init_views=1, phi=3.0, fill_passes=2, w_l2=1.0, w_census=-1.0, p1_frac=0.05,
                p2_frac=0.5, subpixel=1, softmin_tau=0.1, paths=8, edge_threshold=0.0, channels=1, boundless=0,
                fine_radius_far=0, n_lfs=1)


def _case(kind, **kw):
    c = dict(DEFAULTS, kind=kind)
    c.update(kw)
    if c["w_census"] < 0:
        c["w_census"] = 1.0 / (c["census_w"] ** 2 - 1)
    return c


def listed():
    bench = dict(U=9, V=9, H=512, W=512)
    plenoptic = dict(U=15, V=15, H=434, W=625, dmin=-1.5, dmax=1.5, coarse_labels=64, fine_labels=301)
    return [
        # the smallest light field: a live preview or a unit of a tiled job; launches and latency
        _case("depth", name="depth-tiny", U=5, V=5, H=64, W=64, census_w=5, dmin=-2.0, dmax=2.0, coarse_labels=32,
              fine_labels=81, fine_radius=5),
        # a small camera's light field, host to host: the call of an application that holds no device memory
        _case("host", name="host-3x3", U=3, V=3, H=376, W=541, dmin=-1.0, dmax=1.0, coarse_labels=32, fine_labels=101,
              subpixel=2),
        # the 9x9 benchmark light field: its initial pass and its cost volume alone, and the whole method
        # with the soft-argmin read-out
        _case("initial", name="initial-9x9", **bench),
        _case("cost", name="cost-9x9", **bench),
        _case("depth", name="depth-9x9", subpixel=2, **bench),
        # a frame of a 4x4 camera array with short windows, the SGM alone over the paper's 16 directions
        _case("sgm", name="sgm-4x4-16", U=4, V=4, H=720, W=1280, census_w=5, dmin=-6.0, dmax=6.0, coarse_labels=64,
              fine_labels=241, fine_radius=8, paths=16),
        # the final map in colour
        _case("final", name="final-9x9-rgb", subpixel=2, channels=3, **bench),
        # a plenoptic camera's image: many views, a narrow baseline; the final map on given windows
        _case("final", name="final-15x15", subpixel=2, **plenoptic),
        # stereo-like row of views, census only, every pixel searching the whole range
        _case("final", name="final-7x1-boundless", U=7, V=1, H=555, W=650, dmin=0.0, dmax=12.0, coarse_labels=64,
              fine_labels=121, fine_radius=5, boundless=1, w_l2=0.0, w_census=1.0, subpixel=2),
        # training: one step on the benchmark light field, and one on a training crop through autograd
        _case("train", name="train-9x9", subpixel=2, **bench),
        _case("autograd", name="autograd-5x5-crop", U=5, V=5, H=160, W=192, census_w=5, dmin=-2.0, dmax=2.0,
              coarse_labels=32, fine_labels=161, fine_radius=12, subpixel=2),
        # serving: several small light fields of mixed odd sizes in one launch
        _case("batch", name="batch-12-small", U=5, V=5, H=251, W=283, dmin=-2.0, dmax=2.0, coarse_labels=32,
              fine_labels=201, fine_radius=10, subpixel=2, n_lfs=12),
    ]


def draw(rng):
    """A case of the same ranges: 3x3 .. 15x15 views (a row of views for boundless search), images of
    48 .. 720 pixels a side (odd ones among them), windows of 11 .. 31 labels of 81 .. 401, grey or colour,
    both census windows, 8 or 16 directions."""
    def log(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    while True:
        kind = rng.choice(("depth", "host", "initial", "cost", "sgm", "final", "final", "train", "autograd", "batch"))
        kw = dict(U=rng.choice((3, 4, 5, 7, 9, 9, 11, 15)), V=rng.choice((3, 4, 5, 7, 9, 9, 11, 15)), H=log(48, 720),
                  W=log(48, 720), census_w=rng.choice((5, 7)), coarse_labels=log(16, 128),
                  fine_radius=rng.randint(5, 15), paths=rng.choice((8, 8, 8, 16)),
                  channels=rng.choice((1, 1, 1, 3)), subpixel=2)
        far = max(kw["U"], kw["V"]) // 2 + 1
        d = round(min(rng.uniform(1.0, 6.0), 20.0 / far), 2)
        kw.update(dmin=-d, dmax=d, fine_labels=2 * log(40, 200) + 1)
        if kind == "final" and rng.random() < 0.3:
            kw.update(V=1, dmin=0.0, dmax=2 * d, boundless=1, w_l2=0.0, w_census=1.0, channels=1,
                      fine_labels=rng.randint(48, 121))
        if kind == "batch":
            kw.update(H=min(kw["H"], 300), W=min(kw["W"], 300), n_lfs=rng.randint(3, 12), channels=1)
        c = _case(kind, **kw)
        n = c["fine_labels"] if c["boundless"] else 2 * c["fine_radius"] + 1
        cells = c["H"] * c["W"] * n * c["n_lfs"]
        if (cells * (c["U"] * c["V"] - 1) * c["channels"] <= (0.5e9 if kind in ("train", "autograd") else 1.2e9)
                and cells * c["paths"] <= 2.5e8 and c["H"] * c["W"] * c["fine_labels"] <= 1.1e8):
            return c


# ------------------------------------------------------------------ inputs
class _Params:
    """A case's method parameters as attributes (what the package's configurations are made from)."""

    def __init__(self, c, H=None, W=None):
        self.__dict__.update({k: v for k, v in c.items() if k not in ("name", "kind", "n_lfs")})
        self.H, self.W = H or c["H"], W or c["W"]
        self.uc, self.vc = (self.U - 1) // 2, (self.V - 1) // 2
        self.N = self.H * self.W


def _params(c):
    """The parameters of each light field of a case (a batch: sizes around the case's)."""
    return [_Params(c, max(32, c["H"] - 13 * (i % 4)), max(32, c["W"] - 17 * (i % 3))) for i in range(c["n_lfs"])]


def _render(p, seed, dev="cuda"):
    """views [V, U, (C,) H, W] float32: eight slanted planes on the Voronoi cells of eight sites, each with a
    blurred noise texture; the nearest plane whose own cell holds the back-projected point is seen."""
    g = torch.Generator(device=dev).manual_seed(int(seed) * 7919 + 17)
    cpu = torch.Generator().manual_seed(int(seed) * 7919 + 17)
    U, V, H, W, C, K = p.U, p.V, p.H, p.W, p.channels, 8
    span, mid = p.dmax - p.dmin, 0.5 * (p.dmin + p.dmax)
    margin = int(math.ceil(max(abs(p.dmin), abs(p.dmax)) * max(U, V))) + 2
    th, tw = H + 2 * margin, W + 2 * margin
    tex = torch.rand(K, C, th, tw, generator=g, device=dev)
    k3 = torch.tensor([0.25, 0.5, 0.25], device=dev)
    blur = (k3[:, None] * k3[None, :]).view(1, 1, 3, 3)
    pad = torch.nn.functional.pad(tex.view(K * C, 1, th, tw), (1, 1, 1, 1), mode="replicate")
    tex = sum(pad[:, :, i:i + th, j:j + tw] * blur[0, 0, i, j] for i in range(3) for j in range(3)).view(K, C, th * tw)
    r = torch.rand(K, 5, generator=cpu).tolist()
    slope = 0.06 * span
    planes = []
    for a, b, c, sx, sy in r:
        b, c = slope * (2 * b - 1), slope * (2 * c - 1)
        lim = 0.47 * span - 0.5 * (abs(b) + abs(c))
        planes.append((mid + max(-lim, min(lim, 0.85 * span * (a - 0.5))), b, c, sx * W, sy * H))
    sx = torch.tensor([q[3] for q in planes], device=dev).view(-1, 1, 1, 1)
    sy = torch.tensor([q[4] for q in planes], device=dev).view(-1, 1, 1, 1)
    Y, X = torch.meshgrid(torch.arange(H, device=dev, dtype=torch.float32), torch.arange(W, device=dev, dtype=torch.float32),
                          indexing="ij")
    views = torch.empty(V, U, C, H, W, device=dev)
    a = (torch.arange(U, device=dev, dtype=torch.float32) - p.uc).view(U, 1, 1)
    for v in range(V):
        b = float(v - p.vc)
        best = torch.full((U, H, W), -1e30, device=dev)
        img = torch.zeros(U, C, H, W, device=dev)
        for i, (d0, kx, ky, _, _) in enumerate(planes):
            kx, ky = kx / W, ky / H
            k0 = d0 - kx * 0.5 * (W - 1) - ky * 0.5 * (H - 1)
            m00, m01, m10, m11 = 1.0 + a * kx, a * ky, b * kx, 1.0 + b * ky
            r0, r1 = X - a * k0, Y - b * k0
            det = m00 * m11 - m01 * m10
            x, y = (m11 * r0 - m01 * r1) / det, (m00 * r1 - m10 * r0) / det
            own = (x - sx[i]) ** 2 + (y - sy[i]) ** 2
            inside = torch.ones_like(x, dtype=torch.bool)
            for j in range(K):
                if j != i:
                    inside &= own <= (x - sx[j]) ** 2 + (y - sy[j]) ** 2
            # a point outside the plane's own cell is seen only where no plane claims the pixel
            rank = torch.where(inside, k0 + kx * x + ky * y, -1e6 - k0 - kx * x - ky * y)
            gx = (x + margin).clamp(0.0, tw - 1.001)
            gy = (y + margin).clamp(0.0, th - 1.001)
            x0, y0 = gx.floor(), gy.floor()
            fx, fy = (gx - x0).unsqueeze(1), (gy - y0).unsqueeze(1)
            q = (y0 * tw + x0).long()
            t = tex[i]
            s00, s10, s01, s11 = (t[:, q + o].transpose(0, 1) for o in (0, 1, tw, tw + 1))
            smp = (1 - fy) * ((1 - fx) * s00 + fx * s10) + fy * ((1 - fx) * s01 + fx * s11)
            take = rank > best
            best = torch.where(take, rank, best)
            img = torch.where(take.unsqueeze(1), smp, img)
        views[v] = img
    views += 0.01 * torch.randn(views.shape, generator=g, device=dev)
    views.clamp_(0.0, 1.0)
    return views if C > 1 else views[:, :, 0].contiguous()


def _explicit_penalties(p):
    """Fixed P1, P2 of the training cases: the fractions of a typical mean cost."""
    mean = (p.U * p.V - 1) * (0.1 * p.w_l2 * math.sqrt(p.channels) + 0.3 * (p.census_w ** 2 - 1) * p.w_census * p.channels)
    return 0.05 * mean, 0.5 * mean


def _target(p, seed):
    """A smooth disparity map that the training cases are pulled to."""
    g = torch.Generator().manual_seed(int(seed) * 104729 + 5)
    a, b, c = (torch.rand(3, generator=g) - 0.5).tolist()
    y, x = torch.meshgrid(torch.linspace(-1, 1, p.H), torch.linspace(-1, 1, p.W), indexing="ij")
    return (0.5 * (p.dmin + p.dmax) + 0.3 * (p.dmax - p.dmin) * (a + b * x + c * y)).reshape(-1)


def _capacity(p, nnz):
    """Slots of the windowed buffers: a program that runs many light fields of one shape sizes them once, with
    twice the regular windows (more where many pixels search the whole range)."""
    row = (min(2 * p.fine_radius + 1, p.fine_labels) + 3) // 4 * 4
    for room in (2.0, 6.0):
        n = int(p.N * row * room) // 4 * 4
        if nnz <= n and not p.boundless:
            return n
    return p.N * ((p.fine_labels + 3) // 4 * 4)


def prepare(case, seed):
    ps = _params(case)
    s = {"kind": case["kind"], "case": case}
    if case["kind"] == "batch":
        views = [_render(p, seed * 31 + i) for i, p in enumerate(ps)]
        s["batch"] = lf.LightFieldBatch(ps, views, branches=4)
        return s
    p = ps[0]
    views = _render(p, seed)
    s["views"] = views
    if case["kind"] == "host":
        s["views"] = views.cpu().pin_memory()
        s["disp"] = torch.empty(p.N).pin_memory()
        s["L"] = lf.LightFieldDepth(p)
        return s
    L = s["L"] = lf.LightFieldDepth(p)
    if case["kind"] in ("depth", "initial"):
        if case["kind"] == "depth":
            s["disp"] = torch.empty(p.N, device="cuda")
            s["label"] = torch.empty(p.N, dtype=torch.int32, device="cuda")
        return s
    n = _capacity(p, L.initial(views, want_nnz=True))
    s["cost"], s["agg"] = torch.zeros(n, device="cuda"), torch.zeros(n, device="cuda")
    if case["kind"] == "sgm":
        lf.lfsgm_cost_volume(L.h, views, L.lo, L.cnt, L.off, s["cost"])
    if case["kind"] in ("train", "autograd"):
        s["P"] = _explicit_penalties(p)
        s["target"] = _target(p, seed).cuda()
        if case["kind"] == "train":
            s["gcost"], s["gviews"] = torch.zeros(n, device="cuda"), torch.empty_like(views)
            s["gp"] = torch.zeros(2, device="cuda")
        else:
            views.requires_grad_(True)
            s["P"] = [torch.tensor(v, dtype=torch.float32, device="cuda", requires_grad=True) for v in s["P"]]
    return s


def run(s):
    kind = s["kind"]
    if kind == "batch":
        return {"disp": list(s["batch"].run())}
    L, views = s["L"], s["views"]
    if kind == "depth":
        lf.lfsgm_depth(L.h, views, s["disp"], s["label"])
        # the label is the read-out's integer part: it goes with the parabola's read-out only
        return {"disp": s["disp"], "label": s["label"]} if s["case"]["subpixel"] == 1 else {"disp": s["disp"]}
    if kind == "host":
        lf.lfsgm_depth_host(L.h, views, s["disp"])
        return {"disp": s["disp"]}
    if kind == "initial":
        L.initial(views)
        return {"lo": L.lo, "cnt": L.cnt, "off": L.off, "dinit": L.dinit}
    cost, agg = s["cost"], s["agg"]
    if kind == "cost":
        lf.lfsgm_cost_volume(L.h, views, L.lo, L.cnt, L.off, cost)
        return {"cost": cost}
    if kind == "sgm":
        lf.lfsgm_sgm_aggregate(L.h, cost, L.lo, L.cnt, L.off, -1.0, -1.0, agg)
        return {"agg": agg}
    if kind == "final":
        lf.lfsgm_cost_volume(L.h, views, L.lo, L.cnt, L.off, cost)
        lf.lfsgm_sgm_aggregate(L.h, cost, L.lo, L.cnt, L.off, -1.0, -1.0, agg)
        lf.lfsgm_wta_subpixel(L.h, agg, L.lo, L.cnt, L.off, None, L.disp)
        return {"cost": cost, "agg": agg, "disp": L.disp}
    if kind == "train":
        P1, P2 = s["P"]
        lf.lfsgm_cost_volume(L.h, views, L.lo, L.cnt, L.off, cost)
        lf.lfsgm_sgm_aggregate_record(L.h, cost, L.lo, L.cnt, L.off, P1, P2, agg)
        lf.lfsgm_wta_subpixel(L.h, agg, L.lo, L.cnt, L.off, None, L.disp)
        gdisp = (L.disp - s["target"]) * (2.0 / L.N)
        gp = s["gp"]
        lf.lfsgm_backward_recorded(L.h, views, cost, agg, L.lo, L.cnt, L.off, P1, P2, gdisp, s["gcost"], gp[0:1],
                                   gp[1:2], s["gviews"])
        return {"disp": L.disp, "agg": agg, "gcost": s["gcost"], "gP": gp, "gviews": s["gviews"]}
    disp = lf.depth_from_views(views, s["P"][0], s["P"][1], L)
    loss = ((disp - s["target"]) ** 2).mean()
    gv, g1, g2 = torch.autograd.grad(loss, [views, s["P"][0], s["P"][1]])
    return {"disp": disp.detach(), "loss": loss.detach(), "gviews": gv, "gP1": g1, "gP2": g2}


def work(case):
    """Bytes: views read, windows read or written, and the windowed volumes that the call takes or gives, once
    each.  Operations: the coarse matching's Hamming distances and SGM steps, six operations per bilinear
    sample and channel, nine per SGM cell and direction, twice the forward's for the gradients."""
    total = {"bytes": 0.0, "flops": 0.0}
    for p in _params(case):
        kind, nv = case["kind"], p.U * p.V
        n = p.fine_labels if p.boundless else min(2 * p.fine_radius + 1, p.fine_labels)
        cells = float(p.N) * n
        view_bytes = 4.0 * nv * p.channels * p.N
        arm_views, arms = (p.U - 1) + (p.V - 1), (2 if p.U > 1 else 0) + (2 if p.V > 1 else 0)
        coarse = 0.0 if p.boundless else float(p.N) * p.coarse_labels * (2 * arm_views * p.channels + 9 * p.paths * arms)
        samples = (0.0 if p.w_l2 == 0 else 6.0) * cells * (nv - 1) * p.channels + 2.0 * cells * (nv - 1) * p.channels
        sgm = 9.0 * cells * p.paths
        win = 16.0 * p.N
        by, fl = {
            "depth": (view_bytes + 8.0 * p.N, coarse + samples + sgm),
            "host": (view_bytes + 4.0 * p.N, coarse + samples + sgm),
            "batch": (view_bytes + 4.0 * p.N, coarse + samples + sgm),
            "initial": (4.0 * (1 + arm_views) * p.channels * p.N + win + 4.0 * p.N, coarse),
            "cost": (view_bytes + win + 4.0 * cells, samples),
            "sgm": (win + 8.0 * cells, sgm),
            "final": (view_bytes + win + 8.0 * cells + 4.0 * p.N, samples + sgm),
            "train": (2 * view_bytes + win + 8.0 * cells + 8.0 * p.N, 3 * (samples + sgm)),
            "autograd": (2 * view_bytes + win + 8.0 * p.N, 3 * (samples + sgm)),
        }[kind]
        total["bytes"] += by
        total["flops"] += fl
    return total


# ------------------------------------------------------------------ the outputs in 64 bits
_DIRS = ((1, 0), (-1, 0), (0, 1), (0, -1), (1, 1), (-1, -1), (1, -1), (-1, 1), (2, 1), (-2, -1), (2, -1), (-2, 1),
         (1, 2), (-1, -2), (1, -2), (-1, 2))


def _shift(a, d):
    s = a * d
    r = round(2.0 * s)
    if abs(2.0 * s - r) <= 2e-9:
        s = 0.5 * r
    o = math.floor(s)
    return o, s - o, math.floor(s + 0.5)


def _census(img, w):
    """Census words (int64) of img [..., H, W]: bit k is centre > neighbour k, clamped at the border."""
    H, W = img.shape[-2:]
    h, k = w // 2, 0
    ys, xs = torch.arange(H, device=img.device), torch.arange(W, device=img.device)
    out = torch.zeros(img.shape, dtype=torch.int64, device=img.device)
    for dy in range(-h, h + 1):
        rows = img[..., (ys + dy).clamp(0, H - 1), :]
        for dx in range(-h, h + 1):
            if dx or dy:
                out |= (img > rows[..., (xs + dx).clamp(0, W - 1)]).long() << k
                k += 1
    return out


def _popcount(w):
    w = w - ((w >> 1) & 0x5555555555555555)
    w = (w & 0x3333333333333333) + ((w >> 2) & 0x3333333333333333)
    w = (w + (w >> 4)) & 0x0F0F0F0F0F0F0F0F
    w = w + (w >> 8)
    w = w + (w >> 16)
    return (w + (w >> 32)) & 0x7F


def _sgm(cost, P1, P2, paths):
    """Sum over the directions of the path costs of cost [A, H, W, L] (absent labels: a large value or inf);
    P1, P2 numbers or tensors that broadcast over [A, W, L]."""
    A, H, W, K = cost.shape
    big = math.inf if cost.dtype.is_floating_point else 1 << 28

    def step(c, prev, sx):
        # prev: the path costs of the predecessors' row, moved by sx columns; path starts keep c
        if sx:
            fill = torch.full_like(prev[:, :abs(sx)], 0)
            prev = torch.cat((fill, prev[:, :-sx]), 1) if sx > 0 else torch.cat((prev[:, -sx:], fill), 1)
        edge = torch.full_like(prev[..., :1], big)
        m = prev.min(-1, keepdim=True).values
        near = torch.minimum(torch.cat((edge, prev[..., :-1]), -1), torch.cat((prev[..., 1:], edge), -1)) + P1
        new = c + (torch.minimum(torch.minimum(prev, near), m + P2) - m)
        if sx > 0:
            new = torch.cat((c[:, :sx], new[:, sx:]), 1)
        elif sx < 0:
            new = torch.cat((new[:, :sx], c[:, sx:]), 1)
        return new

    total = None
    for dx, dy in _DIRS[:paths]:
        if dy:
            rows = [None] * H
            for y in (range(H) if dy > 0 else range(H - 1, -1, -1)):
                q = y - dy
                rows[y] = cost[:, y] if not 0 <= q < H or abs(dx) >= W else step(cost[:, y], rows[q], dx)
            one = torch.stack(rows, 1)
        else:
            cols = [None] * W
            for x in (range(W) if dx > 0 else range(W - 1, -1, -1)):
                cols[x] = cost[:, :, x] if not 0 <= x - dx < W else step(cost[:, :, x], cols[x - dx], 0)
            one = torch.stack(cols, 2)
        total = one if total is None else total + one
    return total


def _initial(p, views):
    """(lo, cnt, dinit) of the initial pass, all in integers."""
    dev, H, W = views.device, p.H, p.W
    lo = torch.zeros(p.N, dtype=torch.int64, device=dev)
    cnt = torch.full((p.N,), p.fine_labels, dtype=torch.int64, device=dev)
    if p.boundless:
        return lo, cnt, torch.full((p.N,), math.nan, device=dev, dtype=torch.float64)
    v5 = views.view(p.V, p.U, p.channels, H, W)
    ys, xs = torch.arange(H, device=dev), torch.arange(W, device=dev)
    arms = [[(p.uc, v) for v in range(p.vc - 1, -1, -1)], [(p.uc, v) for v in range(p.vc + 1, p.V)],
            [(u, p.vc) for u in range(p.uc - 1, -1, -1)], [(u, p.vc) for u in range(p.uc + 1, p.U)]]
    ref = _census(v5[p.vc, p.uc], p.census_w)
    step = (p.dmax - p.dmin) / (p.coarse_labels - 1)
    costs = []
    for arm in arms:
        if not arm:
            continue
        cost = torch.zeros(H, W, p.coarse_labels, dtype=torch.int32, device=dev)
        for u, v in arm:
            cen, last, h = _census(v5[v, u], p.census_w), None, None
            for k in range(p.coarse_labels):
                d = p.dmin + k * step
                n = _shift(u - p.uc, d)[2], _shift(v - p.vc, d)[2]
                if n != last:
                    at = cen[:, (ys + n[1]).clamp(0, H - 1)][:, :, (xs + n[0]).clamp(0, W - 1)]
                    h, last = _popcount(ref ^ at).sum(0).int(), n
                cost[..., k] += h
        costs.append(cost)
    cost = torch.stack(costs)
    mean = cost.sum((1, 2, 3)).double() / (p.N * p.coarse_labels)
    P1 = (p.p1_frac * mean + 0.5).floor().clamp(min=1)
    P2 = torch.maximum((p.p2_frac * mean + 0.5).floor(), P1)
    agg = _sgm(cost, P1.int().view(-1, 1, 1), P2.int().view(-1, 1, 1), p.paths)
    best = (agg * 256 + torch.arange(p.coarse_labels, device=dev, dtype=torch.int32)).min(-1).values % 256
    best = best.view(len(costs), -1).long() * 8
    F, ok = best[0], torch.ones(p.N, dtype=torch.bool, device=dev)
    for b in best[1:]:
        ok &= (F - b).abs().double() < 8.0 * p.phi
        F = torch.where(ok, (F + b) // 2, F)
    F = torch.where(ok, F, -1).view(H, W)
    none = 1 << 40
    for _ in range(p.fill_passes):
        q = torch.full((H + 2, W + 2), none, dtype=torch.int64, device=dev)
        q[1:-1, 1:-1] = torch.where(F >= 0, F, none)
        near = torch.stack([q[1 + i:1 + i + H, 1 + j:1 + j + W] for i in (-1, 0, 1) for j in (-1, 0, 1) if i or j])
        near = near.sort(0).values
        n = (near < none).sum(0)
        med = near.gather(0, ((n - 1).clamp(min=0) // 2).unsqueeze(0))[0]
        F = torch.where((F < 0) & (n > 0), med, F)
    F = F.reshape(-1)
    den = 8 * (p.coarse_labels - 1)
    gc = (2 * F * (p.fine_labels - 1) + den) // (2 * den)
    a, b = (gc - p.fine_radius).clamp(min=0), (gc + p.fine_radius).clamp(max=p.fine_labels - 1)
    lo = torch.where(F < 0, lo, a)
    cnt = torch.where(F < 0, cnt, b - a + 1)
    return lo, cnt, torch.where(F < 0, math.nan, 0.125 * F.double())


class _Cells:
    """The windows' cells: their place in the padded rows, their pixel and label."""

    def __init__(self, p, lo, cnt):
        dev = lo.device
        rows = (cnt + 3) // 4 * 4
        self.off = torch.zeros(p.N + 1, dtype=torch.int64, device=dev)
        self.off[1:] = rows.cumsum(0)
        self.size = _capacity(p, int(self.off[-1]))
        self.pix = torch.repeat_interleave(torch.arange(p.N, device=dev), cnt)
        j = torch.arange(self.pix.numel(), device=dev) - (cnt.cumsum(0) - cnt)[self.pix]
        self.lab, self.at = lo[self.pix] + j, self.off[self.pix] + j

    def flat(self, v):
        return torch.zeros(self.size, dtype=v.dtype, device=v.device).index_copy(0, self.at, v)

    def dense(self, v, p):
        d = torch.full((p.N * p.fine_labels,), math.inf, dtype=v.dtype, device=v.device)
        return d.index_copy(0, self.pix * p.fine_labels + self.lab, v).view(1, p.H, p.W, p.fine_labels)

    def of_dense(self, d, p):
        return d.reshape(-1)[self.pix * p.fine_labels + self.lab]


def _taps(p, u, v, dev):
    t = []
    for g in range(p.fine_labels):
        d = p.dmin + g * ((p.dmax - p.dmin) / (p.fine_labels - 1))
        x, y = _shift(u - p.uc, d), _shift(v - p.vc, d)
        t.append((x[0], y[0], x[2], y[2], x[1], y[1]))
    t = torch.tensor(t, dtype=torch.float64, device=dev)
    return [t[:, i].long() for i in range(4)] + [t[:, 4], t[:, 5]]


def _l2(p, img, ref, taps, cells, x, y):
    """The l2 distances of one view at the cells; img, ref: [C, N] in 64 bits."""
    ox, oy, _, _, fx, fy = (t[cells.lab] for t in taps)
    xa, xb = (x + ox).clamp(0, p.W - 1), (x + ox + 1).clamp(0, p.W - 1)
    ya, yb = (y + oy).clamp(0, p.H - 1) * p.W, (y + oy + 1).clamp(0, p.H - 1) * p.W
    at = lambda q: img.index_select(1, q)  # noqa: E731
    s = (1 - fy) * ((1 - fx) * at(ya + xa) + fx * at(ya + xb)) + fy * ((1 - fx) * at(yb + xa) + fx * at(yb + xb))
    d = ref.index_select(1, cells.pix) - s
    return d[0].abs() if p.channels == 1 else torch.linalg.vector_norm(d, dim=0)


def _cost(p, views, cells):
    v5 = views.view(p.V, p.U, p.channels, p.H, p.W)
    x, y = cells.pix % p.W, cells.pix // p.W
    ref = v5[p.vc, p.uc].double().view(p.channels, -1)
    cref = _census(v5[p.vc, p.uc], p.census_w).view(p.channels, -1)
    sl2 = torch.zeros(cells.pix.numel(), dtype=torch.float64, device=views.device)
    sc = torch.zeros_like(sl2)
    for v in range(p.V):
        for u in range(p.U):
            if u == p.uc and v == p.vc:
                continue
            taps = _taps(p, u, v, views.device)
            if p.w_l2:
                sl2 += _l2(p, v5[v, u].double().view(p.channels, -1), ref, taps, cells, x, y)
            q = (y + taps[3][cells.lab]).clamp(0, p.H - 1) * p.W + (x + taps[2][cells.lab]).clamp(0, p.W - 1)
            cen = _census(v5[v, u], p.census_w).view(p.channels, -1)
            for c in range(p.channels):
                sc += _popcount(cref[c][cells.pix] ^ cen[c][q])
    return p.w_l2 * sl2 + p.w_census * sc


def _readout(p, dense):
    """The disparities of the aggregated cost [N, G] (inf: absent): parabola or soft-argmin."""
    step = (p.dmax - p.dmin) / (p.fine_labels - 1)
    g = torch.arange(p.fine_labels, device=dense.device, dtype=torch.float64)
    m, b = dense.min(1)
    if p.subpixel == 2:
        w = torch.exp((m[:, None] - dense) / p.softmin_tau)
        return p.dmin + step * (w * g).sum(1) / w.sum(1), b
    cnt = torch.isfinite(dense).sum(1)
    lower = dense.gather(1, (b - 1).clamp(min=0)[:, None])[:, 0]
    upper = dense.gather(1, (b + 1).clamp(max=p.fine_labels - 1)[:, None])[:, 0]
    inner = (cnt >= 5) & (b > 0) & (b < p.fine_labels - 1) & torch.isfinite(lower) & torch.isfinite(upper)
    den = (lower - m) + (upper - m)
    ok = inner & (den > 0)
    delta = torch.where(ok, (lower - upper) / (2 * torch.where(ok, den, 1.0)), 0.0)
    return p.dmin + step * (b.double() + torch.where(ok, delta, 0.0)), b


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for i, p in enumerate(_params(case)):
            views = _render(p, seed * 31 + i)
            lo, cnt, _ = _initial(p, views)
            cells = _Cells(p, lo, cnt)
            cost = _cost(p, views, cells)
            mean = cost.mean()
            agg = _sgm(cells.dense(cost, p), p.p1_frac * mean, p.p2_frac * mean, p.paths)
            out.append(_readout(p, agg.view(p.N, -1))[0])
        return {"disp": out}
    p = _params(case)[0]
    views = _render(p, seed)
    lo, cnt, dinit = _initial(p, views)
    cells = _Cells(p, lo, cnt)
    if kind == "initial":
        return {"lo": None, "cnt": None, "off": None, "dinit": dinit}
    cost = _cost(p, views, cells)
    if kind == "cost":
        return {"cost": cells.flat(cost)}
    if kind not in ("train", "autograd"):
        mean = cost.mean()
        agg = _sgm(cells.dense(cost, p), p.p1_frac * mean, p.p2_frac * mean, p.paths)
        flat = cells.flat(cells.of_dense(agg, p))
        if kind == "sgm":
            return {"agg": flat}
        disp, _ = _readout(p, agg.view(p.N, -1))
        if kind == "final":
            return {"cost": cells.flat(cost), "agg": flat, "disp": disp}
        return {"disp": disp, "label": None} if p.subpixel == 1 else {"disp": disp}
    # gradients: the aggregate and read-out by autograd, then the l2 term view by view
    P1, P2 = (torch.tensor(float(torch.tensor(v, dtype=torch.float32)), dtype=torch.float64, device=views.device,
                           requires_grad=True) for v in _explicit_penalties(p))
    cost.requires_grad_(True)
    agg = _sgm(cells.dense(cost, p), P1, P2, p.paths)
    disp, _ = _readout(p, agg.view(p.N, -1))
    loss = ((disp - _target(p, seed).to(views.device).double()) ** 2).mean()
    gcost, g1, g2 = torch.autograd.grad(loss, [cost, P1, P2])
    flat = cells.flat(cells.of_dense(agg.detach(), p))
    del agg
    v5 = views.view(p.V, p.U, p.channels, p.H, p.W)
    x, y = cells.pix % p.W, cells.pix // p.W
    gviews = torch.zeros(v5.shape, dtype=torch.float64, device=views.device)
    ref = v5[p.vc, p.uc].double().view(p.channels, -1).requires_grad_(True)
    for v in range(p.V):
        for u in range(p.U):
            if u == p.uc and v == p.vc:
                continue
            img = v5[v, u].double().view(p.channels, -1).requires_grad_(True)
            term = (gcost * p.w_l2 * _l2(p, img, ref, _taps(p, u, v, views.device), cells, x, y)).sum()
            gi, gr = torch.autograd.grad(term, [img, ref])
            gviews[v, u] += gi.view(p.channels, p.H, p.W)
            gviews[p.vc, p.uc] += gr.view(p.channels, p.H, p.W)
    gviews = gviews.view(views.shape)
    if kind == "train":
        return {"disp": disp.detach(), "agg": flat, "gcost": cells.flat(gcost), "gP": torch.stack((g1, g2)),
                "gviews": gviews}
    return {"disp": disp.detach(), "loss": loss.detach(), "gviews": gviews, "gP1": g1, "gP2": g2}
