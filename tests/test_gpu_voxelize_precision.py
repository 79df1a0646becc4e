"""Level-1 clusters whose points lie close together in a large voxel, near the
sensor: their sums lose no more than FP64 sums of the offsets do, whatever the
voxel's size.  Lengths on both sides of a warp's and of a piece's points."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS = np.finfo(np.float64).eps


@pytest.fixture(scope="module")
def mm():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2608_14266_gb300 as mm
    assert torch.cuda.is_available()
    return mm


@pytest.mark.parametrize("voxel", [0.5, 2.0, 40.0, 1000.0])
@pytest.mark.parametrize("spread", [(1e-4, 1e-4, 1e-4), (0.02, 0.02, 0.02), (0.2, 0.2, 0.001), (0.1, 1e-6, 0.05)])
def test_small_clusters_in_large_voxels(mm, voxel, spread):
    """Scans of one cluster each, in a voxel of its own (poses move them there).
    Tolerance: the recursive-summation bound of shifted sums over chunks of 32
    points, k eps of the sums of the terms' sizes with k = min(n, 32) + n / 32 + 8,
    the final operations included; a mean also rounds to its own last bit."""
    rng = np.random.default_rng(int(voxel * 8))
    lens = [1, 2, 3, 5, 10, 31, 33, 100, 191, 192, 193, 1000, 1024, 1025, 5000, 40000]
    centre = rng.uniform(-0.3, 0.3, (len(lens), 3))  # metres from the sensor
    centre[::3] *= 1e-3
    pts = [c + rng.uniform(-0.5, 0.5, (n, 3)) * spread for c, n in zip(centre, lens)]
    spo = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    poses = np.tile(np.concatenate([np.eye(3).ravel(), np.zeros(3)]), (len(lens), 1))
    poses[:, 9:] = voxel * np.array([0.5, 0.5, 0.5]) - centre
    poses[:, 9] += voxel * np.arange(len(lens))
    got = mm.voxelize(spo, np.concatenate(pts), poses, voxel)
    np.testing.assert_array_equal(got["obs_scan"], np.arange(len(lens)))
    np.testing.assert_array_equal(got["agg"][:, 9], lens)
    for row, p in zip(got["agg"], pts):
        x = p.astype(np.longdouble)
        n, m = len(x), x.mean(0)
        d, o = x - m, np.abs(x - x[0])
        k = (min(n, 32) + n / 32 + 8) * EPS
        assert np.all(np.abs(row[6:9] - m) <= k * o.sum(0) / n + EPS * np.abs(m)), n
        q = 0
        for a in range(3):
            for b in range(a, 3):
                size = (o[:, a] * o[:, b]).sum() + o[:, a].sum() * o[:, b].sum() / n
                assert abs(row[q] - (d[:, a] * d[:, b]).sum()) <= k * size, (n, a, b)
                q += 1


def test_many_runs_of_close_points(mm):
    """Enough such runs for a lane each, and in batches of few of them for four:
    the same bits, and the bound above (all entries of a chunk of 32 points and
    fewer) for a sample."""
    rng = np.random.default_rng(11)
    side = 320  # 102,400 voxels of 2 m in the plane of the sensor
    lens = rng.integers(2, 24, side * side)
    lens[rng.integers(0, side * side, 50)] = 70
    i = np.arange(side * side)
    centre = np.stack([(i % side - side / 2 + 0.5) * 2.0, (i // side - side / 2 + 0.5) * 2.0,
                       rng.uniform(0.3, 0.6, side * side)], 1)
    pts = np.repeat(centre, lens, axis=0) + rng.uniform(-0.5, 0.5, (lens.sum(), 3)) * [0.5, 0.5, 1e-3]
    n = len(pts)
    spo = np.array([0, n], dtype=np.int64)
    pose = np.concatenate([np.eye(3).ravel(), np.zeros(3)])[None]
    import torch
    args = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (spo, pts, pose)]
    got = {k: v.cpu().numpy() for k, v in mm.voxelize(*args, 2.0, out="device").items() if hasattr(v, "cpu")}
    index = np.floor(centre / 2.0).astype(np.int64)
    order = np.lexsort((index[:, 2], index[:, 1], index[:, 0]))
    np.testing.assert_array_equal(got["agg"][:, 9], lens[order])
    # scans of one row each, in batches of a few
    rows = np.concatenate([[0], np.cumsum(lens)])[::side]
    poses = np.repeat(pose, side, axis=0)
    small = mm.voxelize(rows.astype(np.int64), pts, poses, 2.0, batch_points=20000)
    assert small["batches"] > 50
    np.testing.assert_array_equal(small["agg"], got["agg"])
    start = np.concatenate([[0], np.cumsum(lens)])
    for r in rng.integers(0, len(lens), 300):
        v = order[r]
        x = pts[start[v] : start[v + 1]].astype(np.longdouble)
        m, o = x.mean(0), np.abs(x - x[0])
        d, k = x - m, (min(len(x), 32) + len(x) / 32 + 8) * EPS
        q = 0
        for a in range(3):
            for b in range(a, 3):
                size = (o[:, a] * o[:, b]).sum() + o[:, a].sum() * o[:, b].sum() / len(x)
                assert abs(got["agg"][r, q] - (d[:, a] * d[:, b]).sum()) <= k * size, (r, a, b)
                q += 1
