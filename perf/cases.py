"""Timed cases of the DeGraF + RLOF + EPIC framework.

Each case is one call, or one short chain of calls, that a program using this package
makes, through its public entry points:

* ``pair``     one device-resident frame pair: key-points, both pyramids, tracking
               (``PairTracker.run``), with the support radius, motion model, storage
               type and cross-based support as options;
* ``batch``    many pairs of mixed sizes and steps in one call (``BatchTracker.run``);
* ``host``     host frames in, host results out (``HostPairTracker.run``);
* ``front``    key-points with their exact window sums and the pyramid with gradients
               (``detect``, ``build_pyramid``), as a program that tracks later calls them;
* ``fb``       key-points, pyramids and the forward-backward filter (``track_fb``);
* ``epic``     dense flow from sparse matches (``epic_interpolate``);
* ``dense``    the whole DeGraF-Flow method (``DenseFlow.run``) with the global-motion prior;
* ``adjoint``  forward and backward through ``DeGraFDetect`` and ``RLOFTrack``.

Frames are uint8 textures (64 Gaussian blobs and three octaves of value noise) drawn
from the seed. Scene "shift": frame 2 is frame 1 translated by a few pixels plus
N(0, 2) noise, as in neighbouring frames of slow motion. Scene "drive": radial
expansion reaching ``reach`` pixels at the corners plus three rectangles with their own
translations, the shape of a driving sequence.
"""
import math

import numpy as np
import torch

import paper_1901_09971_gb300 as dgf

BATCH_SIZES = ((640, 480), (1024, 436), (1242, 375), (1280, 720))
BATCH_STEPS = (2, 3, 4, 6)


# ------------------------------------------------------------------ the cases


def listed():
    return [
        # a small pair on its own: launches and latency
        {"name": "pair_256x128", "kind": "pair", "scene": "shift", "W": 256, "H": 128, "win": 8, "step": 4,
         "levels": 3, "radius": 4, "model": 4, "f16": False, "tau": 0.0},
        # a driving frame pair, dense key-points, large motion
        {"name": "pair_1242x375", "kind": "pair", "scene": "drive", "W": 1242, "H": 375, "win": 7, "step": 3,
         "levels": 5, "radius": 5, "model": 4, "f16": False, "tau": 0.0},
        # a recorded sequence processed offline: 16 pairs of mixed sizes in one call
        {"name": "batch_16_mixed", "kind": "batch", "scene": "shift", "pairs": 16, "mix": 3000, "win": 8,
         "levels": 3, "radius": 4, "model": 4, "f16": False},
        # a camera loop: frames arrive in host memory, results leave to it; half storage
        {"name": "host_640x480_f16", "kind": "host", "scene": "shift", "W": 640, "H": 480, "win": 8, "step": 3,
         "levels": 3, "radius": 4, "model": 4, "f16": True},
        # the front end on an odd-sized frame, with the exact sums
        {"name": "front_1279x719", "kind": "front", "scene": "shift", "W": 1279, "H": 719, "win": 8, "step": 4,
         "levels": 4, "f16": False},
        # a wide support without the illumination terms, ragged size
        {"name": "pair_641x479_r7", "kind": "pair", "scene": "shift", "W": 641, "H": 479, "win": 5, "step": 5,
         "levels": 3, "radius": 7, "model": 2, "f16": False, "tau": 0.0},
        # the adaptive cross-based support
        {"name": "pair_1242x375_cross", "kind": "pair", "scene": "drive", "W": 1242, "H": 375, "win": 8, "step": 4,
         "levels": 4, "radius": 4, "model": 4, "f16": False, "tau": 20.0},
        # consistency-checked matches
        {"name": "fb_1024x436", "kind": "fb", "scene": "shift", "W": 1024, "H": 436, "win": 8, "step": 4,
         "levels": 4, "radius": 5, "model": 4, "f16": False},
        # interpolation of a small frame with a short neighbourhood
        {"name": "epic_256x128", "kind": "epic", "scene": "drive", "W": 256, "H": 128, "step": 4, "k": 32,
         "affine": True},
        # interpolation of the driving frame's dense matches (k = 128 as in the paper)
        {"name": "epic_1242x375", "kind": "epic", "scene": "drive", "W": 1242, "H": 375, "step": 3, "k": 128,
         "affine": True},
        # the whole method
        {"name": "dense_1242x375", "kind": "dense", "scene": "drive", "W": 1242, "H": 375, "win": 7, "step": 3,
         "levels": 5, "radius": 5, "model": 4, "extra": 0, "k": 128},
        # a learning loop: forward and backward for both frames
        {"name": "adjoint_1242x375", "kind": "adjoint", "scene": "shift", "W": 1242, "H": 375, "win": 8, "step": 4,
         "levels": 3, "radius": 4, "model": 4, "f16": False},
    ]


def _size(rng, lo=160, hi=1400):
    """A frame size, spread over the logarithm, odd ones among them."""
    W = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    H = max(96, int(round(W * rng.choice((0.3, 0.45, 0.5625, 0.75)))))
    return W, H


def draw(rng):
    kind = rng.choice(("pair", "pair", "pair", "batch", "host", "front", "fb", "epic", "epic", "dense", "adjoint"))
    scene = rng.choice(("shift", "drive"))
    radius = rng.choice((4, 4, 5, 5, 3, 7))
    model = rng.choice((4, 4, 4, 2))
    f16 = rng.random() < 0.25
    step = rng.choice((3, 4, 4, 5, 6, 9))
    win = rng.choice((3, 5, 7, 8, 8, 8, 11))
    W, H = _size(rng)
    levels = rng.choice((2, 3, 4) if min(W, H) >= 256 else (2, 3) if min(W, H) >= 128 else (1, 2))
    base = {"kind": kind, "scene": scene}
    if kind == "batch":
        return {**base, "pairs": rng.randint(2, 8), "mix": rng.randint(1, 1 << 20), "win": 8, "levels": 3,
                "radius": rng.choice((4, 4, 5)), "model": 4, "f16": f16}
    base.update(W=W, H=H)
    if kind == "front":
        return {**base, "win": win, "step": step, "levels": levels, "f16": f16}
    if kind == "epic":
        return {**base, "step": rng.choice((3, 4, 5, 7, 10)), "k": rng.choice((5, 16, 32, 64, 128, 128, 200)),
                "affine": rng.random() < 0.85}
    if kind == "dense":
        return {**base, "win": win, "step": step, "levels": levels, "radius": rng.choice((4, 5)), "model": 4,
                "extra": rng.choice((0, 1)) if min(W, H) >> (levels + 1) >= 12 else 0, "k": rng.choice((64, 128))}
    base.update(win=win, step=step, levels=levels, radius=radius, model=model, f16=f16)
    if kind == "pair":
        base["tau"] = rng.choice((0.0, 0.0, 0.0, 15.0, 30.0))
    return base


# ----------------------------------------------------------------- the inputs


def _dev():
    return torch.device("cuda")


class _Texture:
    """A continuous random texture: blobs and value noise, separable in x and y."""

    def __init__(self, rng, W, H):
        self.cx, self.cy = rng.uniform(0, W, 64), rng.uniform(0, H, 64)
        self.sigma, self.amp = rng.uniform(W / 64, W / 8, 64), rng.uniform(-1, 1, 64)
        self.octaves = []
        for spacing, amp in ((32.0, 1.0), (16.0, 0.5), (8.0, 0.25)):
            nx, ny = int(math.ceil(W / spacing)) + 12, int(math.ceil(H / spacing)) + 12
            self.octaves.append((spacing, amp, rng.uniform(-1, 1, (ny, nx))))

    @staticmethod
    def _weights(at, spacing, n):
        u = at / spacing + 5
        i = torch.floor(u).long().clamp(0, n - 2)
        t = (u - i).clamp(0, 1)
        s = (t * t * (3 - 2 * t)).unsqueeze(1)
        w = torch.zeros(at.numel(), n, dtype=torch.float64, device=at.device)
        w.scatter_(1, i.unsqueeze(1), 1 - s)
        return w.scatter_(1, i.unsqueeze(1) + 1, s)

    def at(self, xs, ys):
        """The texture's values on the grid ys x xs."""
        def t(v):
            return torch.from_numpy(np.asarray(v)).to(xs.device)

        two = 2 * t(self.sigma) ** 2
        ex = torch.exp(-((xs[:, None] - t(self.cx)) ** 2) / two)
        ey = torch.exp(-((ys[:, None] - t(self.cy)) ** 2) / two)
        v = (ey * t(self.amp)) @ ex.T
        for spacing, amp, lattice in self.octaves:
            ny, nx = lattice.shape
            v = v + amp * (self._weights(ys, spacing, ny) @ t(lattice) @ self._weights(xs, spacing, nx).T)
        return v


def _bytes(v):
    return torch.round(v).clamp(0, 255).to(torch.uint8).contiguous()


def _frames(scene, W, H, seed):
    """Two uint8 frames on the GPU and the true flow of frame 1's pixels [H, W, 2]."""
    rng, dev = np.random.default_rng(seed), _dev()
    noise = torch.Generator(device=dev)
    noise.manual_seed(int(seed))
    xs = torch.arange(W, dtype=torch.float64, device=dev)
    ys = torch.arange(H, dtype=torch.float64, device=dev)
    tex = _Texture(rng, W, H)
    raw1 = tex.at(xs, ys)
    if scene == "shift":
        tx, ty = rng.uniform(-6, 6), rng.uniform(-3, 3)
        raw2 = tex.at(xs - tx, ys - ty)
        flow = torch.empty(H, W, 2, dtype=torch.float64, device=dev)
        flow[..., 0], flow[..., 1] = tx, ty
    else:
        cx, cy = (W - 1) / 2, (H - 1) / 2
        g = min(150.0, 0.12 * W) / math.hypot(cx, cy)
        raw2 = tex.at(cx + (xs - cx) / (1 + g), cy + (ys - cy) / (1 + g))
        flow = torch.stack(torch.broadcast_tensors(g * (xs - cx)[None, :], g * (ys - cy)[:, None]), dim=-1).clone()
        for _ in range(3):
            rw, rh = int(rng.integers(W // 15, W // 4)), int(rng.integers(H // 9, H * 2 // 5))
            x0, y0 = int(rng.integers(0, W - rw)), int(rng.integers(0, H - rh))
            tx, ty = rng.uniform(-1, 1, 2) * min(60.0, 0.05 * W)
            own = _Texture(rng, rw, rh)
            raw1[y0:y0 + rh, x0:x0 + rw] = own.at(xs[:rw], ys[:rh])
            flow[y0:y0 + rh, x0:x0 + rw, 0], flow[y0:y0 + rh, x0:x0 + rw, 1] = tx, ty
            cover = (((ys >= y0 + ty) & (ys < y0 + ty + rh))[:, None] & ((xs >= x0 + tx) & (xs < x0 + tx + rw))[None, :])
            raw2 = torch.where(cover, own.at(xs - (x0 + tx), ys - (y0 + ty)), raw2)
    lo, hi = raw1.min(), raw1.max()
    scale = 224 / (hi - lo).clamp_min(1e-12)
    extra = torch.randn(H, W, dtype=torch.float64, device=dev, generator=noise) * 2
    return _bytes(16 + scale * (raw1 - lo)), _bytes(16 + scale * (raw2 - lo) + extra), flow.float()


def _params(c):
    return dgf.RlofParams(levels=c["levels"], radius=c["radius"], model=c["model"],
                          storage=dgf.F16 if c.get("f16") else dgf.F32, cross_tau=c.get("tau", 0.0))


def _specs(c):
    rng = np.random.default_rng(c["mix"])
    out = []
    for _ in range(c["pairs"]):
        W, H = BATCH_SIZES[int(rng.integers(0, 4))]
        out.append((W, H, c["win"], BATCH_STEPS[int(rng.integers(0, 4))]))
    return out


def _matches(c, flow, seed):
    """Sparse matches as tracking leaves them: key-points around the centres of a grid of
    7-pixel windows, true flow with small errors, a few gross outliers, lost patches."""
    W, H, step, dev = c["W"], c["H"], c["step"], _dev()
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed) + 77)
    u = torch.arange((W - 7) // step + 1, device=dev) * step
    v = torch.arange((H - 7) // step + 1, device=dev) * step
    pts = torch.stack(torch.broadcast_tensors(u[None, :], v[:, None]), dim=-1).reshape(-1, 2).float() + 3
    n = pts.shape[0]

    def rand(*shape):
        return torch.rand(*shape, device=dev, generator=g)

    pts = (pts + rand(n, 2) - 0.5).contiguous()
    at = pts.round().long()
    f = flow[at[:, 1], at[:, 0]] + 0.1 * torch.randn(n, 2, device=dev, generator=g)
    f = torch.where(rand(n, 1) < 0.02, f + 20 * (rand(n, 2) - 0.5), f)
    status = torch.where(rand(n) < 0.03, 4, 0)
    status = torch.where(rand(n) < 0.05, 2, status)
    spots = rand(6, 3)
    for k in range(6):
        r = 0.02 * W + 0.05 * W * spots[k, 2]
        near = (pts[:, 0] - spots[k, 0] * W) ** 2 + (pts[:, 1] - spots[k, 1] * H) ** 2 < r * r
        status = torch.where(near, 1, status)
    f = torch.where(((status == 0) | (status == 4))[:, None], f, 0.0)
    return pts, f.float().contiguous(), status.to(torch.uint8).contiguous()


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "batch":
        specs = _specs(c)
        frames = [_frames(c["scene"], W, H, 1000 * (seed % 100003) + i)[:2] for i, (W, H, _, _) in enumerate(specs)]
        tracker = dgf.BatchTracker(specs, _params(c), _dev())
        tracker.bind([f[0] for f in frames], [f[1] for f in frames])
        return {"kind": kind, "tracker": tracker}
    W, H = c["W"], c["H"]
    f1, f2, flow = _frames(c["scene"], W, H, seed)
    s = {"kind": kind, "case": c, "f1": f1, "f2": f2}
    if kind == "pair":
        s["tracker"] = dgf.PairTracker(W, H, c["win"], c["step"], _params(c), _dev())
    elif kind == "host":
        s["tracker"] = dgf.HostPairTracker(W, H, c["win"], c["step"], _params(c), _dev())
        s["f1"], s["f2"] = f1.cpu().pin_memory(), f2.cpu().pin_memory()
    elif kind == "front":
        layout = dgf.pyramid_layout(W, H, c["levels"], dgf.F16 if c["f16"] else dgf.F32, True)
        s["storage"] = layout["storage"]
        s["pyramid"] = torch.empty(layout["bytes"], dtype=torch.uint8, device=_dev())
        s["planes"] = [list(p) for p in dgf.pyramid_planes(s["pyramid"], layout)]
    elif kind == "fb":
        s["params"] = _params(c)
    elif kind == "epic":
        s["matches"] = _matches(c, flow, seed)
        s["params"] = dgf.EpicParams(k=c["k"], model=1 if c["affine"] else 0)
        n = s["matches"][0].shape[0]
        s["workspace"] = torch.empty(dgf.epic_workspace_bytes(W, H, n), dtype=torch.uint8, device=_dev())
    elif kind == "dense":
        s["flow"] = dgf.DenseFlow(W, H, c["win"], c["step"], _params(c), gm=dgf.GmParams(extra_levels=c["extra"]),
                                  epic=dgf.EpicParams(k=c["k"]), device=_dev())
    else:
        g = torch.Generator(device=_dev())
        g.manual_seed(int(seed) + 5)
        n = dgf.degraf_count(W, H, c["win"], c["step"])
        s["params"] = _params(c)
        s["f1"], s["f2"] = f1.float().requires_grad_(), f2.float().requires_grad_()
        s["up_pts"] = torch.randn(n, 2, device=_dev(), generator=g)
        s["up_flow"] = torch.randn(n, 2, device=_dev(), generator=g)
    return s


# ------------------------------------------------------------------- one pass


def run(s):
    kind = s["kind"]
    if kind == "batch":
        return [list(v) for v in s["tracker"].run()]
    if kind in ("pair", "host"):
        return list(s["tracker"].run(s["f1"], s["f2"]))
    c = s["case"]
    if kind == "front":
        pts, sums = dgf.detect(s["f1"], c["win"], c["step"], with_sums=True)
        dgf.build_pyramid(s["f1"], c["levels"], s["storage"], True, out=s["pyramid"])
        return {"pts": pts, "sums": sums, "planes": s["planes"]}
    if kind == "fb":
        p = s["params"]
        pts = dgf.detect(s["f1"], c["win"], c["step"])
        p1 = dgf.build_pyramid(s["f1"], p.levels, p.storage, True)
        p2 = dgf.build_pyramid(s["f2"], p.levels, p.storage, True)
        return [pts, *dgf.track_fb(p1, p2, c["W"], c["H"], pts, p, 1.0)]
    if kind == "epic":
        return dgf.epic_interpolate(s["f1"], *s["matches"], s["params"], workspace=s["workspace"])
    if kind == "dense":
        dense, sparse = s["flow"].run(s["f1"], s["f2"])
        return [dense, *sparse]
    pts = dgf.DeGraFDetect.apply(s["f1"], c["win"], c["step"])
    (g_pts,) = torch.autograd.grad(pts, s["f1"], s["up_pts"])
    flow, status = dgf.RLOFTrack.apply(s["f1"], s["f2"], pts.detach(), s["params"])
    g1, g2 = torch.autograd.grad(flow, (s["f1"], s["f2"]), s["up_flow"])
    return [pts.detach(), g_pts, flow.detach(), status, g1, g2]


# ------------------------------------------------------------ work of one pass


def _count(W, H, win, step):
    return ((W - win) // step + 1) * ((H - win) // step + 1)


def _pixels(W, H, levels):
    return sum((W >> l) * (H >> l) for l in range(levels))


def _track_flops(n, c):
    """Tracking of n points: per sample and step 41 (gain and offset) or 24 operations
    and per level 33 for the template, at the steps a level takes on these scenes."""
    steps = 13 if c["scene"] == "drive" else 7
    samples = (2 * c["radius"] + 1) ** 2
    return float(n) * c["levels"] * samples * (33 + steps * (41 if c["model"] == 4 else 24))


def _epic_flops(W, H, n, k):
    """Per pixel the edge cost, four relaxations and the model; per seed k settled
    neighbours of a six-neighbour graph and their 12 weighted sums."""
    return 60.0 * W * H + float(n) * k * (6 * 8 + 50)


def work(case):
    c, kind = case, case["kind"]
    if kind == "batch":
        b = f = 0.0
        for W, H, win, step in _specs(c):
            n = _count(W, H, win, step)
            b += 2 * W * H + 18 * n
            f += _track_flops(n, c) + 12.0 * W * H
        return {"bytes": b, "flops": f}
    W, H = c["W"], c["H"]
    n = _count(W, H, c.get("win", 7), c["step"])
    es = 2 if c.get("f16") else 4
    if kind == "front":
        return {"bytes": W * H + 24 * n + 3 * es * _pixels(W, H, c["levels"]),
                "flops": 12.0 * _pixels(W, H, c["levels"]) + 6.0 * n * c["win"] ** 2}
    if kind == "epic":
        return {"bytes": W * H + 17 * n + 8 * W * H, "flops": _epic_flops(W, H, n, c["k"])}
    front = 12.0 * W * H
    if kind == "pair" or kind == "host":
        return {"bytes": 2 * W * H + 18 * n, "flops": front + _track_flops(n, c)}
    if kind == "fb":
        return {"bytes": 2 * W * H + 21 * n, "flops": front + 2 * _track_flops(n, c)}
    if kind == "dense":
        return {"bytes": 2 * W * H + 17 * n + 8 * W * H,
                "flops": front + 1.25 * _track_flops(n, c) + _epic_flops(W, H, n, c["k"])}
    return {"bytes": 8 * W * H + 33 * n + 12 * W * H,
            "flops": front + _track_flops(n, c) + 150.0 * n * (2 * c["radius"] + 1) ** 2}


# -------------------------------------------------------- outputs in 64 bits


def _box(v, win, step):
    """Sums of v [H, W] over every win x win window, exactly (int64)."""
    s = torch.zeros(v.shape[0] + 1, v.shape[1] + 1, dtype=torch.int64, device=v.device)
    s[1:, 1:] = v.cumsum(0).cumsum(1)
    a = s[win:, win:] - s[:-win, win:] - s[win:, :-win] + s[:-win, :-win]
    return a[::step, ::step]


def _exact_points(frame, win, step):
    """Key-points (float64) and their sums: the darker- or brighter-weighted centroid of
    each window, whichever weight sum is larger."""
    I = frame.long()
    H, W = I.shape
    x = torch.arange(W, device=I.device)[None, :]
    y = torch.arange(H, device=I.device)[:, None]
    S = _box(I, win, step)
    u = torch.arange(S.shape[1], device=I.device)[None, :] * step
    v = torch.arange(S.shape[0], device=I.device)[:, None] * step
    X, Y = _box(I * x, win, step) - u * S, _box(I * y, win, step) - v * S
    m = torch.nn.functional.max_pool2d(frame.double()[None, None], win, stride=1)[0, 0, ::step, ::step].long()
    n, moment = win * win, win * (win * (win - 1) // 2)
    Sn, Xn, Yn = n * (1 + m) - S, (1 + m) * moment - X, (1 + m) * moment - Y
    neg = Sn > S
    den = torch.where(neg, Sn, S).double()
    px = u + torch.where(neg, Xn, X).double() / den
    py = v + torch.where(neg, Yn, Y).double() / den
    return torch.stack((px, py), -1).reshape(-1, 2), torch.stack((S, X, Y, m), -1).reshape(-1, 4)


def _exact_planes(frame, levels):
    out, I = [], frame.double()
    for l in range(levels):
        p = torch.nn.functional.pad(I[None, None], (1, 1, 1, 1), mode="replicate")[0, 0]
        d, s = p[:, 2:] - p[:, :-2], p[:, :-2] + 2 * p[:, 1:-1] + p[:, 2:]
        out.append([I, (d[:-2] + 2 * d[1:-1] + d[2:]) / 8, (s[2:] - s[:-2]) / 8])
        h, w = I.shape[0] // 2, I.shape[1] // 2
        if l + 1 < levels:
            I = I[:2 * h, :2 * w].reshape(h, 2, w, 2).mean((1, 3))
    return out


def _exact_point_gradient(frame, win, step, up):
    """Gradient of sum(up * key-points) with respect to the frame: of the chosen centroid,
    whose inverted weights 1 + m - I follow the window's first maximum."""
    H, W = frame.shape
    cols = torch.nn.functional.unfold(frame.double()[None, None], win, stride=step)[0].T  # [windows, win * win]
    j = torch.arange(win, device=frame.device).repeat(win).double()
    i = torch.arange(win, device=frame.device).repeat_interleave(win).double()
    m, S = cols.max(1).values, cols.sum(1)
    first = (cols == m[:, None]).double().argmax(1)
    Sn = win * win * (1 + m) - S
    neg = Sn > S
    wgt = torch.where(neg[:, None], 1 + m[:, None] - cols, cols)
    den = wgt.sum(1)
    arm = (up[:, :1] * (j - ((wgt * j).sum(1) / den)[:, None]) + up[:, 1:] * (i - ((wgt * i).sum(1) / den)[:, None]))
    arm = arm / den[:, None]
    g = torch.where(neg[:, None], -arm, arm)
    g.scatter_add_(1, first[:, None], torch.where(neg, arm.sum(1), 0.0)[:, None])
    return torch.nn.functional.fold(g.T[None], (H, W), win, stride=step)[0, 0]


def _exact_epic(c, frame, pts, flow, status, k, affine):
    """The interpolation in whole-number distances and 64-bit fits: edge costs from the
    Sobel magnitudes, geodesic cells of the matches, the cells' graph, each match's k
    nearest in it, a weighted affine fit (or mean), every pixel by its match's model."""
    W, H, dev, n = c["W"], c["H"], _dev(), pts.shape[0]
    p = torch.nn.functional.pad(frame.double()[None, None], (1, 1, 1, 1), mode="replicate")[0, 0].long()
    d, s = p[:, 2:] - p[:, :-2], p[:, :-2] + 2 * p[:, 1:-1] + p[:, 2:]
    C = 4 + (d[:-2] + 2 * d[1:-1] + d[2:]).abs() + (s[2:] - s[:-2]).abs()
    none = torch.iinfo(torch.int64).max
    key = torch.full((H * W,), none, dtype=torch.int64, device=dev)
    ok = (status == 0) | (status == 4)
    at = torch.floor(pts + 0.5).long()
    pix = at[:, 1].clamp(0, H - 1) * W + at[:, 0].clamp(0, W - 1)
    ids = torch.arange(n, device=dev)
    key.scatter_reduce_(0, pix[ok], ids[ok], "amin")
    seed = torch.zeros(n, dtype=torch.bool, device=dev)
    seed[key[key < none]] = True
    key = key.reshape(H, W)
    wx, wy = (C[:, 1:] + C[:, :-1]) << 24, (C[1:] + C[:-1]) << 24
    far = none - (1 << 50)
    key = key.clamp_max(far)
    while True:  # min-plus relaxation of (distance, match) to its fixed point
        old = key.clone()
        for _ in range(16):
            key[:, 1:] = torch.minimum(key[:, 1:], key[:, :-1] + wx)
            key[:, :-1] = torch.minimum(key[:, :-1], key[:, 1:] + wx)
            key[1:] = torch.minimum(key[1:], key[:-1] + wy)
            key[:-1] = torch.minimum(key[:-1], key[1:] + wy)
        if torch.equal(old, key):
            break
    lab, dist = key & ((1 << 24) - 1), key >> 24
    a = torch.cat((lab[:, 1:].reshape(-1), lab[1:].reshape(-1)))
    b = torch.cat((lab[:, :-1].reshape(-1), lab[:-1].reshape(-1)))
    w = torch.cat(((dist[:, 1:] + dist[:, :-1] + (wx >> 24)).reshape(-1),
                   (dist[1:] + dist[:-1] + (wy >> 24)).reshape(-1)))
    a, b, w = torch.cat((a, b)), torch.cat((b, a)), torch.cat((w, w))
    edge, back = torch.unique((a * n + b)[a != b], return_inverse=True)
    ew = torch.full((edge.numel(),), none, dtype=torch.int64, device=dev).scatter_reduce_(0, back, w[a != b], "amin")
    ea, eb = edge // n, edge % n
    models = torch.zeros(n, 6, dtype=torch.float64, device=dev)
    sources = ids[seed]
    big = 1 << 40
    for rows in sources.split(512):
        D = torch.full((rows.numel(), n), big, dtype=torch.int64, device=dev)
        D[torch.arange(rows.numel(), device=dev), rows] = 0
        while True:
            N = D.clone()
            N.scatter_reduce_(1, eb[None].expand(rows.numel(), -1), D[:, ea] + ew, "amin")
            if torch.equal(N, D):
                break
            D = N
        rank = torch.where(D < big, (D << 20) + ids, none)
        near = rank.topk(min(k, n), dim=1, largest=False, sorted=True).values
        have = near < none
        t, dt = torch.where(have, near & ((1 << 20) - 1), 0), torch.where(have, near >> 20, 0)
        wt = torch.where(have, torch.exp(-0.1 / 8.0 * dt.double()), 0.0)
        v = torch.cat((pts[t].double() - pts[rows].double()[:, None], torch.ones_like(wt)[..., None]), -1)
        f = flow[t].double()
        M = torch.einsum("sk,ski,skj->sij", wt, v, v)
        r = torch.einsum("sk,ski,skj->sij", wt, v, f)
        m22 = M[:, 2, 2]
        mean = M[:, :2, 2] / m22[:, None]
        cov = M[:, :2, :2] / m22[:, None, None] - mean[:, :, None] * mean[:, None, :]
        half = 0.5 * (cov[:, 0, 0] - cov[:, 1, 1])
        lam = 0.5 * (cov[:, 0, 0] + cov[:, 1, 1]) - torch.sqrt(half ** 2 + cov[:, 0, 1] ** 2)
        use = (lam >= 1.0) & (have.sum(1) >= 3) & affine
        eye = torch.eye(3, dtype=torch.float64, device=dev)
        sol = torch.linalg.solve(torch.where(use[:, None, None], M, eye), r)
        models[rows, 4:] = torch.where(use[:, None], sol[:, 2], r[:, 2] / m22[:, None])
        models[rows, 0:2] = torch.where(use[:, None], sol[:, :2, 0], 0.0)
        models[rows, 2:4] = torch.where(use[:, None], sol[:, :2, 1], 0.0)
    m, q = models[lab], pts[lab].double()
    dx = torch.arange(W, device=dev).double()[None, :] - q[..., 0]
    dy = torch.arange(H, device=dev).double()[:, None] - q[..., 1]
    return torch.stack((m[..., 0] * dx + m[..., 1] * dy + m[..., 4], m[..., 2] * dx + m[..., 3] * dy + m[..., 5]), -1)


def exact(case, seed):
    """Key-points, sums, planes, key-point gradients and (for frames of up to 6000 matches)
    the dense field in 64 bits. The tracked flow has no such value: its iteration stops
    at an iteration cap, a step size and lost-point tests, so the last bits of the
    arithmetic decide where some of its points end."""
    c, kind = case, case["kind"]
    if kind == "batch":
        pts = []
        for i, (W, H, win, step) in enumerate(_specs(c)):
            f1 = _frames(c["scene"], W, H, 1000 * (seed % 100003) + i)[0]
            pts.append(_exact_points(f1, win, step)[0])
        none = [None] * len(pts)
        return [pts, none, none, none]
    f1, _, flow = _frames(c["scene"], c["W"], c["H"], seed)
    if kind == "epic":
        pts, f, status = _matches(c, flow, seed)
        return _exact_epic(c, f1, pts, f, status, c["k"], c["affine"]) if pts.shape[0] <= 6000 else None
    pts, sums = _exact_points(f1, c["win"], c["step"])
    if kind == "front":
        return {"pts": pts, "sums": sums, "planes": _exact_planes(f1, c["levels"])}
    if kind == "pair":
        return [pts, None, None, None]
    if kind == "host":
        return [pts, None, None]
    if kind == "fb":
        return [pts, None, None, None]
    if kind == "dense":
        return [None, pts, None, None]
    g = torch.Generator(device=_dev())
    g.manual_seed(int(seed) + 5)
    up = torch.randn(pts.shape[0], 2, device=_dev(), generator=g).double()
    return [pts, _exact_point_gradient(f1, c["win"], c["step"], up), None, None, None, None]
