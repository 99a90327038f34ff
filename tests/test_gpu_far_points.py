"""Tracking of points far outside the frame, infinite or NaN: any position may be given.
A point whose coordinates leave the range of int is handled as one that is merely far
away in the same direction, and none changes another's result."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

FAR, NEAR = 3e9, 1e5  # beyond 2^31, and well within it


@pytest.mark.parametrize("radius,lanes,model,tau,f16", [(4, 8, 4, 0.0, False), (5, 8, 4, 0.0, False), (4, 8, 2, 0.0, False),
                                                        (5, 8, 4, 15.0, False), (5, 8, 4, 0.0, True), (4, 16, 4, 0.0, False),
                                                        (3, 0, 4, 0.0, False), (7, 0, 2, 15.0, True)])
def test_points_anywhere(radius, lanes, model, tau, f16):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1901_09971_gb300 as dgf
    p = synth.make_pair(1, size=(201, 133))
    prm = dgf.RlofParams(levels=3, radius=radius, model=model, cross_tau=tau, storage=dgf.F16 if f16 else dgf.F32, min_eig=0.05)
    pyr = [dgf.build_pyramid(torch.from_numpy(f).cuda(), 3, prm.storage, True) for f in (p.I1, p.I2)]
    own = dgf.detect(torch.from_numpy(p.I1).cuda(), 8, 9)

    def track(pts):
        return [t.cpu().numpy() for t in dgf.track(*pyr, p.W, p.H, pts, prm, with_iters=True)]

    def outside(d):
        return [(sx * d if sx else 71.25, sy * d if sy else 55.5) for sx in (-1, 0, 1) for sy in (-1, 0, 1) if sx or sy]

    inf, nan = float("inf"), float("nan")
    odd = [(inf, 20.0), (20.0, -inf), (-inf, -inf), (inf, inf), (nan, 20.0), (20.0, nan), (nan, inf)]
    prev = dgf.set_lanes(lanes)
    try:
        ref = track(own)
        res = {}
        for name, extra in (("far", outside(FAR)), ("huge", outside(3e38)), ("near", outside(NEAR)), ("odd", odd)):
            extra = torch.tensor(extra, dtype=torch.float32, device="cuda")
            mixed = own.clone()
            where = torch.arange(extra.shape[0], device="cuda") * 5 + 2
            mixed[where] = extra
            got = track(mixed)
            keep = np.ones(own.shape[0], bool)
            keep[where.cpu().numpy()] = False
            for g, r in zip(got, ref):
                np.testing.assert_array_equal(g[keep].view(np.uint8), r[keep].view(np.uint8))
            res[name] = [g[~keep] for g in got]
            assert (res[name][0] == 0).all() and np.isin(res[name][1], (1, 2)).all()  # lost, flow 0
        for name in ("far", "huge"):
            for g, r in zip(res[name], res["near"]):
                np.testing.assert_array_equal(g, r)
        assert (res["odd"][1] == 1).all()
    finally:
        dgf.set_lanes(prev)
