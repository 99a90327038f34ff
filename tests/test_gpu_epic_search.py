"""GPU parity of EPIC's neighbourhood search and fits against the oracle at the edges of
its layouts: neighbourhood sizes around the selection's and the sort's widths, ties at
the last neighbour, more matches than one launch's sums hold, weights past the table's
end. Indices and distances are exact integers; models within 1e-9 and the dense field
within 1e-4 px, as for every EPIC case."""
import numpy as np
import pytest
import torch

from test_gpu_epic import assert_parity, dgf, run_both  # noqa: F401
from test_oracle_epic import random_matches, textured

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [2, 31, 32, 33, 63, 64, 65, 127, 129, 160, 161, 255])
def test_neighbourhood_sizes(dgf, k):  # noqa: F811
    W, H = 96, 64
    img = textured(W, H, k)
    pts, flow, status = random_matches(W, H, 500, k)
    g, o = run_both(dgf, img, pts, flow, status, k=k)
    assert_parity(g, o)


@pytest.mark.parametrize("k,cost_gain", [(24, 0), (140, 0), (24, 1)])
def test_ties_at_the_last_neighbour(dgf, k, cost_gain):  # noqa: F811
    """A regular grid on a flat frame: many seeds at the same distance, so the index
    decides which of them are kept."""
    img = np.full((60, 80), 90, np.uint8)
    y, x = np.mgrid[2:60:4, 2:80:4]
    pts = np.stack([x.ravel(), y.ravel()], 1).astype(np.float64)
    flow = np.random.default_rng(k).normal(0, 1, pts.shape)
    g, o = run_both(dgf, img, pts, flow, np.zeros(len(pts), np.uint8), k=k, cost_gain=cost_gain)
    assert_parity(g, o)


@pytest.mark.parametrize("copies", [1, 3])
def test_more_matches_than_one_launch_holds(dgf, copies):  # noqa: F811
    """A match at every pixel (and several at each): beyond W H / 3 holders the searches
    run in further launches."""
    W, H = 47, 31
    img = textured(W, H, 21)
    y, x = np.mgrid[0:H, 0:W]
    pts = np.tile(np.stack([x.ravel(), y.ravel()], 1).astype(np.float64), (copies, 1))
    rng = np.random.default_rng(22)
    status = np.where(rng.random(len(pts)) < 0.05, 1, 0).astype(np.uint8)
    g, o = run_both(dgf, img, pts, rng.normal(0, 1, pts.shape), status, k=20)
    assert (g["fit_kind"] > 0).sum() > W * H // 3
    assert_parity(g, o)


def test_weights_past_the_table(dgf):  # noqa: F811
    """Costs of 4,096 a pixel put most neighbours past the table of weights; the slow
    decay keeps their weights in the fit."""
    W, H = 120, 90
    img = textured(W, H, 31)
    pts, flow, status = random_matches(W, H, 250, 31)
    g, o = run_both(dgf, img, pts, flow, status, k=40, cost_base=4096, cost_gain=2, a=0.05)
    assert np.median(g["knn_dist"][g["knn_dist"] > 0]) > 16384
    assert_parity(g, o)


def test_calls_in_sequence_share_a_workspace(dgf):  # noqa: F811
    """Launches of a call overlap with the kernels before them: calls of other sizes in a
    row on one dirty workspace, and the same in a captured graph, give the bits of calls
    alone on zeroed ones."""
    prm = dgf.EpicParams(k=24)
    sets = []
    for W, H, n in ((256, 128, 1900), (40, 33, 60), (203, 97, 3000), (64, 64, 500)):
        pts, flow, status = random_matches(W, H, n, n)
        sets.append([torch.from_numpy(v).cuda() for v in (textured(W, H, n), pts.astype(np.float32),
                                                          flow.astype(np.float32), status)])
    room = max(dgf.epic_workspace_bytes(s[0].shape[1], s[0].shape[0], len(s[1])) for s in sets)
    alone = []
    for s in sets:
        alone.append(dgf.epic_interpolate(*s, prm, workspace=torch.zeros(room, dtype=torch.uint8, device="cuda")))
        torch.cuda.synchronize()
    ws = torch.full((room,), 0xAB, dtype=torch.uint8, device="cuda")
    outs = [torch.full_like(d, -7.0) for d in alone + alone]

    def run():
        for i, o in enumerate(outs):
            dgf.epic_interpolate(*sets[i % len(sets)], prm, workspace=ws, out=o)

    def check():
        torch.cuda.synchronize()
        for i, o in enumerate(outs):
            assert torch.equal(o, alone[i % len(sets)])
            o.fill_(-7.0)

    run()
    check()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run()
    graph.replay()
    check()
    graph.replay()
    check()
    assert dgf.device_status() == 0
