"""Level-1 clusters of long runs, which are summed in pieces of 1,024 points over
the whole GPU: lengths on both sides of a thread's (192), of a piece and of a
warp's 32 pieces, in host batches that split them, and the offsets that the
integer sums of a piece hold."""
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


def _check(row, pts, size):
    """The recursive-summation bound of shifted sums over chunks of 32 points and
    less, k eps of the sums' size with k = min(n, 32) + n / 32 + 8, offsets of at
    most `size`."""
    x = pts.astype(np.longdouble)
    n, m = len(x), x.mean(0)
    d = x - m
    s = np.array([(d[:, a] * d[:, b]).sum() for a in range(3) for b in range(a, 3)])
    k = (min(n, 32) + n / 32 + 8) * EPS
    assert row[9] == n
    assert np.abs(row[6:9] - m).max() <= k * size + EPS * np.abs(m).max()
    assert np.abs(row[:6] - s).max() <= 2 * k * n * size**2


@pytest.mark.parametrize("batch", [0, 3000, 70000])
def test_lengths(mm, batch):
    rng = np.random.default_rng(3)
    lens = [1, 191, 192, 193, 1023, 1024, 1025, 2048, 2049, 32 * 1024, 32 * 1024 + 1, 70001, 5, 400]
    pts = [rng.uniform(0.0, 1.0, (n, 3)) + [7.0, 3.0, 11.0] for n in lens]
    spo = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    poses = np.tile(np.concatenate([np.eye(3).ravel(), np.full(3, 0.5)]), (len(lens), 1))
    poses[:, 9] += 2.0 * np.arange(len(lens))
    poses[:, 9:] -= [7.0, 3.0, 11.0]
    got = mm.voxelize(spo, np.concatenate(pts), poses, 2.0, batch_points=batch)
    np.testing.assert_array_equal(got["obs_scan"], np.arange(len(lens)))
    for row, p in zip(got["agg"], pts):
        _check(row, p, 1.0)
    again = mm.voxelize(spo, np.concatenate(pts), poses, 2.0, batch_points=batch)
    np.testing.assert_array_equal(got["agg"], again["agg"])


@pytest.mark.parametrize("reach", [2.0 - 2.0**-40, 2.0, 2.01])
@pytest.mark.parametrize("signs", [(1, 1, 1), (-1, -1, -1), (1, -1, 1)])
def test_offsets_at_the_halves_bound(mm, reach, signs):
    """A pose that shrinks the scan sixteenfold leaves offsets of one sign up to the
    2^54 steps that the halves hold (from a first point of 1.75, of 2^-53) inside a
    voxel of 1 m; past them the run takes FP64 sums."""
    p0 = np.array([1.75, 1.5, 1.25])
    lens = [2, 3, 190, 191, 192, 1024, 1025, 8128, 8129]
    pts = [np.concatenate([p0[None], np.tile(p0 + reach * np.array(signs), (n - 1, 1))]) for n in lens]
    spo = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    poses = np.tile(np.concatenate([np.eye(3).ravel() / 16, np.full(3, 0.4)]), (len(lens), 1))
    poses[:, 9] += np.arange(len(lens))
    got = mm.voxelize(spo, np.concatenate(pts), poses, 1.0)
    np.testing.assert_array_equal(got["agg"][:, 9], lens)
    for row, p in zip(got["agg"], pts):
        _check(row, p, reach)
