"""Tracking's short steps against full steps (model 4), bit for bit.

A short step (the right-hand side only, while all residuals have Hampel weight 1) must
give what a full step gives. The two constant sets here give the same weights, bit for
bit: with c = 1e12 the outer factor clamp((c - |r|) / (c - b)) rounds to 1 for every
residual of 8-bit frames, whether b is 8 or 1e11, and a is the same. But the limit up to
which a step may be short is a in one and not positive in the other, so one run takes
short steps wherever they are predicted and the other takes none, in every layout, lane
count and support, with gated points and with start displacements too."""
import numpy as np
import pytest
import torch

import synth

SHORT = dict(hampel_a=8.0, hampel_b=1e11, hampel_c=1e12)
NEVER = dict(hampel_a=8.0, hampel_b=8.0, hampel_c=1e12)


def limit(hampel_a, hampel_b, hampel_c):
    """The largest residual a short step accepts, and the outer factor's constants."""
    f = np.float32
    icb = f(1) / (f(hampel_c) - f(hampel_b))
    hc_icb = f(hampel_c) * icb
    return min(float(f(hampel_a)) * (1 - 1e-6), (float(hc_icb) - 1) / float(icb)), icb, hc_icb


def test_constants():
    """Same weights, different limits."""
    r = np.linspace(0, 1000, 100001).astype(np.float32).astype(np.float64)
    for c, lo, hi in ((SHORT, 7.99, 8.0), (NEVER, -1.0, 0.0)):
        r_in, icb, hc_icb = limit(**c)
        assert lo <= r_in <= hi
        outer = np.clip((float(hc_icb) - r * float(icb)).astype(np.float32), 0, 1)  # a fused multiply-add, clamped
        assert (outer == 1).all()


def test_close_constants():
    """The sets of test_limits_below_a: the outer factor decides, or nothing is left."""
    assert [round(limit(**c)[0], 2) for c in CLOSE] == [0.95, 7.15, 0.0]


CLOSE = (dict(hampel_a=1.0, hampel_b=1.0, hampel_c=2e6), dict(hampel_a=8.0, hampel_b=8.0, hampel_c=3e7),
         dict(hampel_a=1.0, hampel_b=1.0, hampel_c=1e8))


@pytest.fixture(scope="module")
def dgf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1901_09971_gb300 as m
    m.load()
    return m


def frames(config):
    p = synth.make_pair(config, size=(330, 210))
    return p, torch.from_numpy(p.I1).cuda(), torch.from_numpy(p.I2).cuda()


def equal(a, b):
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x.cpu().numpy().view(np.uint8), y.cpu().numpy().view(np.uint8))


@pytest.mark.gpu
@pytest.mark.parametrize("config", [1, 2])
@pytest.mark.parametrize("radius,lanes,tau,f16", [(4, 8, 0.0, False), (5, 8, 0.0, False), (4, 8, 15.0, False), (5, 8, 0.0, True),
                                                  (5, 8, 15.0, True), (4, 16, 0.0, True), (5, 16, 0.0, False), (5, 32, 0.0, False),
                                                  (4, 32, 15.0, False), (1, 0, 0.0, False), (2, 0, 15.0, False), (3, 0, 0.0, False),
                                                  (6, 0, 0.0, True), (7, 0, 15.0, False)])
def test_short_steps_give_the_bits_of_full_steps(dgf, config, radius, lanes, tau, f16):
    p, f1, f2 = frames(config)
    storage = dgf.F16 if f16 else dgf.F32
    pyr = [dgf.build_pyramid(f, 4, storage, True) for f in (f1, f2)]
    low = [dgf.build_pyramid(f, 3, storage, True) for f in (f1, f2)]
    pts = dgf.detect(f1, 8, 5)
    out = []
    prev = dgf.set_lanes(lanes)
    try:
        for c in (SHORT, NEVER):
            prm = dgf.RlofParams(levels=3, radius=radius, cross_tau=tau, storage=storage, **c)
            res = list(dgf.track(*low, p.W, p.H, pts, prm, with_iters=True, with_illum=True))
            assert (res[1] == 0).any()
            # the backward pass leaves out the points that the forward pass lost
            res += dgf.track_fb(*low, p.W, p.H, pts, prm, 1.0)
            # start displacements
            res += dgf.track_gm(*pyr, p.W, p.H, 4, pts, prm, dgf.GmParams(extra_levels=1), with_iters=True, with_illum=True)
            out.append(res)
    finally:
        dgf.set_lanes(prev)
    equal(*out)


@pytest.mark.gpu
def test_some_steps_are_short(dgf):
    """Points of the cases above do meet the condition: their residuals at the result lie
    within the limit, so that the steps near it had all weights 1, and they took several
    steps a level."""
    p, f1, f2 = frames(1)
    prm = dgf.RlofParams(levels=3, radius=4, **SHORT)
    pyr = [dgf.build_pyramid(f, 3, dgf.F32, True) for f in (f1, f2)]
    pts = dgf.detect(f1, 8, 5)
    flow, status, iters, illum = dgf.track(*pyr, p.W, p.H, pts, prm, with_iters=True, with_illum=True)
    k = torch.arange(-4, 5, device="cuda", dtype=torch.float64)
    ky, kx = torch.meshgrid(k, k, indexing="ij")

    def sample(img, at):
        x, y = at[:, 0, None, None] + kx, at[:, 1, None, None] + ky
        x0, y0 = x.floor(), y.floor()
        ax, ay = x - x0, y - y0
        tap = lambda i, j: img.double()[(y0.long() + j).clamp(0, p.H - 1), (x0.long() + i).clamp(0, p.W - 1)]
        return (1 - ay) * ((1 - ax) * tap(0, 0) + ax * tap(1, 0)) + ay * ((1 - ax) * tap(0, 1) + ax * tap(1, 1))

    m, c = illum.double()[:, 0, None, None], illum.double()[:, 1, None, None]
    r = sample(f2, pts.double() + flow.double()) - (1 + m) * sample(f1, pts.double()) - c
    inside = (r.abs().amax((1, 2)) < 7.9) & (status == 0) & (iters >= 3 * 3)
    assert int(inside.sum()) > pts.shape[0] // 10


@pytest.mark.gpu
@pytest.mark.parametrize("constants", range(len(CLOSE)))
@pytest.mark.parametrize("radius,lanes", [(4, 8), (5, 8), (4, 16)])
def test_limits_below_a(dgf, constants, radius, lanes):
    """Constants where the outer factor leaves 1 before a, or at once: the results do not
    depend on which points share a warp, and so not on which steps are short."""
    p, f1, f2 = frames(1)
    prm = dgf.RlofParams(levels=3, radius=radius, **CLOSE[constants])
    pyr = [dgf.build_pyramid(f, 3, dgf.F32, True) for f in (f1, f2)]
    pts = dgf.detect(f1, 8, 5)
    n = pts.shape[0]
    prev = dgf.set_lanes(lanes)
    try:
        track = lambda order: dgf.track(*pyr, p.W, p.H, pts[order].contiguous(), prm, with_iters=True, with_illum=True)
        ref = track(torch.arange(n, device="cuda"))
        for seed in range(3):
            order = torch.from_numpy(np.random.default_rng(seed).permutation(n)).cuda()
            equal(track(order), [r[order] for r in ref])
    finally:
        dgf.set_lanes(prev)
