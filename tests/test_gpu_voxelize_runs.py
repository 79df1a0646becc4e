"""The level-1 clusters of ba_voxelize where their kernel branches: runs
around the length a warp takes over and around the 32 x 254 points of its sums,
the integer and the FP64 path of the voxel indices, coordinates near zero (where the fixed-point step is set by the voxel, not by
the coordinate), few runs (pools of 64) and many (pools of 128)."""
import numpy as np
import pytest

import oracle

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


def _pose(t=(0.0, 0.0, 0.0)):
    return np.concatenate([np.eye(3).ravel(), np.asarray(t, dtype=np.float64)])


@pytest.mark.parametrize("length", [1, 2, 24, 191, 192, 193, 400, 32 * 254, 32 * 254 + 1, 20000])
@pytest.mark.parametrize("offset", [0.0, 1e-9, 57.3])
def test_run_lengths(mm, length, offset):
    """Three scans of one voxel each: `length`, 1 and 7 points within 0.5 m.
    Tolerance against sums in extended precision, per point an offset's
    rounding (2^-53 of the diagonal), per entry the final operations (a few eps
    of the sums' size)."""
    rng = np.random.default_rng(length)
    lens = [length, 1, 7]
    pts = [rng.uniform(0.0, 0.5, (n, 3)) + offset * np.array([1.0, 0.5, 0.0]) for n in lens]
    spo = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    # each scan's points moved into a voxel of its own by the pose
    poses = np.stack([_pose(np.array([0.0, 0.0, 4.0 * j]) - offset * np.array([1.0, 0.5, 0.0])) for j in range(3)])
    P = np.concatenate(pts)
    ref = oracle.voxelize(spo, P, poses, 2.0)
    got = mm.voxelize(spo, P, poses, 2.0)
    for k in ("voxel_off", "obs_scan", "level", "index"):
        np.testing.assert_array_equal(got[k], ref[k])
    np.testing.assert_array_equal(got["agg"][:, 9], ref["agg"][:, 9])
    whole = all(len(np.unique(np.floor((p + q[9:]) / 2.0), axis=0)) == 1 for p, q in zip(pts, poses))
    assert whole or offset != 0.0  # (rounding of p + t may split a scan over two voxels)
    if not whole:
        return
    diag = 2.0 * np.sqrt(3.0)
    for row, j in zip(got["agg"], got["obs_scan"]):
        x = pts[j].astype(np.longdouble)
        n, m = len(x), x.mean(0)
        d = x - m
        s = np.array([(d[:, a] * d[:, b]).sum() for a in range(3) for b in range(a, 3)])
        assert np.abs(row[6:9] - m).max() <= EPS * diag + 2 * EPS * np.abs(m).max()
        size = float(((x - x[0]) ** 2).sum())
        assert np.abs(row[:6] - s).max() <= n * EPS * diag + 4 * EPS * size


@pytest.mark.parametrize("n", [3000, 450000])
def test_many_short_runs(mm, n):
    """Every point in a run of its own or of a few, on both sides of the pool
    size's line; the structure bit for bit, clusters to the recursive-summation
    bound."""
    rng = np.random.default_rng(n)
    base = rng.uniform(-60.0, 60.0, (n, 3))
    reps = rng.integers(1, 3, n)
    P = np.repeat(base, reps, axis=0) + rng.uniform(0.0, 0.05, (int(reps.sum()), 3))
    spo = np.array([0, len(P) // 3, len(P) // 3, len(P)], dtype=np.int64)
    poses = np.stack([_pose((3.0 * j, -j, 0.25)) for j in range(3)])
    ref = oracle.voxelize(spo, P, poses, 0.3)
    got = mm.voxelize(spo, P, poses, 0.3)
    for k in ("voxel_off", "obs_scan", "level", "index"):
        np.testing.assert_array_equal(got[k], ref[k])
    cnt = ref["agg"][:, 9]
    np.testing.assert_array_equal(got["agg"][:, 9], cnt)
    tol = 2 * (cnt + 1) * EPS * 3 * cnt * 0.3**2
    assert np.all(np.abs(got["agg"][:, :6] - ref["agg"][:, :6]) <= tol[:, None])
    assert np.all(np.abs(got["agg"][:, 6:9] - ref["agg"][:, 6:9]) <= 4 * EPS * (60.0 + cnt[:, None]))


def _rotation(rng):
    q, _ = np.linalg.qr(rng.normal(size=(3, 3)))
    return q if np.linalg.det(q) > 0 else -q


@pytest.mark.parametrize("d", [0.5, 0.3, 1.0, 0.7, 1e-3, 40.0, 1e-5])
@pytest.mark.parametrize("form", ["rotation", "identity", "scaled", "far", "long", "limit", "empty"])
def test_index_paths(mm, d, form):
    """Indices bit for bit (the oracle forms floor(RN(w / d)) in FP64): points
    on, just below and just above voxel faces among random ones; poses with a
    rotation, the identity (faces hit exactly), a matrix larger than the fixed
    point takes, offsets near 2^20 voxels; points past the integer path's range;
    coordinates at zero; scans without points between those with some."""
    rng = np.random.default_rng(5)
    m = 4000
    cells = rng.integers(-300, 300, (m, 3)).astype(np.float64)
    p = np.concatenate([cells * d, np.nextafter(cells * d, np.inf), np.nextafter(cells * d, -np.inf),
                        (cells + 2.0**-16 * rng.normal(size=(m, 3))) * d, rng.uniform(-400, 400, (m, 3)) * d,
                        np.zeros((3, 3)), rng.normal(size=(50, 3)) * 1e-300])
    R, t = np.eye(3), np.zeros(3)
    if form == "rotation":
        R, t = _rotation(rng), rng.uniform(-50, 50, 3) * d
    elif form == "scaled":
        R = 37.0 * _rotation(rng)
    elif form == "far":
        R, t = _rotation(rng), np.array([2.0**20 - 2000, -(2.0**20) + 2000, 12345.678]) * d
    elif form == "long":
        R = _rotation(rng)
        p = np.concatenate([p, rng.uniform(-60000, 60000, (m, 3)) * d])
    elif form == "limit":
        t = np.array([2.0**20 - 402.0, 0.0, -(2.0**20) + 402.0]) * d
    n = len(p)
    poses = np.stack([np.concatenate([R.ravel(), t]), np.concatenate([np.eye(3).ravel(), np.zeros(3)]),
                      np.concatenate([R.ravel(), t + d])])
    spo = np.array([0, n // 2, n // 2 if form == "empty" else n // 2 + 5, n], dtype=np.int64)
    if form == "empty":
        poses = np.repeat(poses, [1, 700, 1], axis=0)
        spo = np.concatenate([[0], np.full(701, n // 2), [n]]).astype(np.int64)
    ref = oracle.voxelize(spo, p, poses, d)
    got = mm.voxelize(spo, p, poses, d)
    for k in ("voxel_off", "obs_scan", "level", "index"):
        np.testing.assert_array_equal(got[k], ref[k])
    np.testing.assert_array_equal(got["agg"][:, 9], ref["agg"][:, 9])


@pytest.mark.parametrize("value", [np.nan, np.inf, 1e300, 2.0**20])
def test_point_outside_the_index_range_is_refused(mm, value):
    p = np.random.default_rng(1).uniform(-5, 5, (5000, 3))
    p[3210, 1] = value
    poses = np.stack([np.concatenate([np.eye(3).ravel(), np.zeros(3)])])
    with pytest.raises(mm.BAError, match="point 3210"):
        mm.voxelize(np.array([0, 5000], dtype=np.int64), p, poses, 1.0)
