"""Tracking's short steps (right-hand sides only while all residuals of a warp's points
have weight 1) give the bits of full steps: which steps are short depends on the points
that share a warp, so a point's results must not change with its neighbours. Every
case tracks the same points in raster order, shuffled (each warp another mix of
converging, oscillating and outlier points) and in short calls that leave a warp's
groups idle, and compares all outputs bit for bit. The Hampel constants cover the usual
ones, knees so close together that the weight-1 range ends before hampel_a, a range that
is empty, and one that no residual leaves (short steps only)."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dgf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1901_09971_gb300 as m
    m.load()
    return m


HAMPEL = {"default": {}, "close": dict(hampel_a=7.9, hampel_b=7.95, hampel_c=8.0),
          "steep": dict(hampel_a=1.0, hampel_b=1.0, hampel_c=500.0), "tiny": dict(hampel_a=1e-6, hampel_b=2.0, hampel_c=9.0),
          "wide": dict(hampel_a=600.0, hampel_b=700.0, hampel_c=800.0)}


@pytest.mark.parametrize("hampel", sorted(HAMPEL))
@pytest.mark.parametrize("radius,lanes,tau,f16", [(4, 8, 0.0, False), (5, 8, 0.0, False), (4, 8, 15.0, False),
                                                  (5, 8, 15.0, True), (4, 16, 0.0, True), (5, 32, 0.0, False),
                                                  (3, 0, 0.0, False), (7, 0, 15.0, False)])
def test_results_do_not_depend_on_the_warp(dgf, hampel, radius, lanes, tau, f16):
    p = synth.make_pair(2, size=(330, 210))
    f1, f2 = torch.from_numpy(p.I1).cuda(), torch.from_numpy(p.I2).cuda()
    prm = dgf.RlofParams(levels=3, radius=radius, cross_tau=tau, storage=dgf.F16 if f16 else dgf.F32, **HAMPEL[hampel])
    p1 = dgf.build_pyramid(f1, 3, prm.storage, True)
    p2 = dgf.build_pyramid(f2, 3, prm.storage, False)
    pts = dgf.detect(f1, 8, 5)
    n = pts.shape[0]

    def track(order):
        out = dgf.track(p1, p2, p.W, p.H, pts[order].contiguous(), prm, with_iters=True, with_illum=True)
        return [t.cpu().numpy() for t in out]

    prev = dgf.set_lanes(lanes)
    try:
        ref = track(torch.arange(n, device="cuda"))
        assert (ref[1] == 0).any() and len(np.unique(ref[2])) > 3
        rng = np.random.default_rng(radius)
        for order in (rng.permutation(n), np.arange(n)[::-1].copy(), *(rng.permutation(n)[:k] for k in (1, 2, 3, 5, 7))):
            got = track(torch.from_numpy(order).cuda())
            for g, r in zip(got, ref):
                np.testing.assert_array_equal(g.view(np.uint8), r[order].view(np.uint8))
    finally:
        dgf.set_lanes(prev)
