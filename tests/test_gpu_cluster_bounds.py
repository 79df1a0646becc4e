"""Point clusters at the bounds of their integer sums: offsets of one sign just
below and above the 2^54 steps that two 27-bit halves hold, chunks of 254 points
joined, and numbers of observations on both sides of a block's 128 and 256 and
of the line between one and two rounds a block (38,912)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS = np.finfo(np.float64).eps
P0 = np.array([1.75, 1.0, 1.0 / 3.0])  # steps of 2^-53: half the last bit of 1.75


@pytest.fixture(scope="module")
def mm():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2608_14266_gb300 as mm
    assert torch.cuda.is_available()
    return mm


def _clusters(mm, po, pts):
    import torch
    out = torch.empty((len(po) - 1, 10), dtype=torch.float64, device="cuda")
    mm.ba_aggregate_points(torch.from_numpy(po).cuda(), torch.from_numpy(pts).cuda(), out)
    torch.cuda.synchronize()
    return out.cpu().numpy()


def _check(got, pts, reach):
    """Against sums in extended precision: the integer sums are exact in steps of
    2^-53, so an entry is off by the rounding of its points to a step (n 2 reach
    2^-53), and by a few roundings of the sums' size."""
    x = pts.astype(np.longdouble)
    n, m = len(x), x.mean(0)
    d = x - m
    s = np.array([(d[:, a] * d[:, b]).sum() for a in range(3) for b in range(a, 3)])
    raw = ((x - x[0]) ** 2).sum()
    assert got[9] == n
    assert np.abs(got[6:9] - m).max() <= 2.0**-52 + 4 * EPS * (2 + reach)
    assert np.abs(got[:6] - s).max() <= n * 2 * reach * 2.0**-52 + 4 * EPS * raw


@pytest.mark.parametrize("length", [2, 127, 253, 254, 255, 508, 509, 16384])
@pytest.mark.parametrize("signs", [(1, 1, 1), (-1, -1, -1), (1, -1, 1)])
@pytest.mark.parametrize("reach", [2 - 2.0**-51, 2.0, 2.01, 1.0])
def test_offsets_of_one_sign(mm, length, signs, reach):
    """Every point but the first at the corner: 2 - 2^-51 is 2^54 - 4 steps (high
    half 2^27 - 1, low half 2^27 - 4), 2 and more go to 128-bit sums."""
    pts = np.tile(P0 + reach * np.array(signs), (length, 1))
    pts[0] = P0
    po = np.array([0, length], dtype=np.int64)
    _check(_clusters(mm, po, pts)[0], pts, reach)


@pytest.mark.parametrize("n_obs", [1, 127, 128, 129, 257, 38912, 38913, 39100])
def test_numbers_of_observations(mm, n_obs):
    rng = np.random.default_rng(n_obs)
    lens = rng.integers(0, 12, n_obs)
    lens[:: max(1, n_obs // 7)] = rng.integers(100, 600, len(lens[:: max(1, n_obs // 7)]))
    po = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    pts = P0 + rng.uniform(-1.5, 1.5, (po[-1], 3))
    pts[po[:-1][lens > 0]] = P0
    got = _clusters(mm, po, pts)
    np.testing.assert_array_equal(got[:, 9], lens)
    np.testing.assert_array_equal(got[lens == 0], 0.0)
    pick = np.unique(np.concatenate([np.arange(min(n_obs, 300)), np.arange(max(0, n_obs - 300), n_obs),
                                     np.flatnonzero(lens > 12)]))
    for o in pick[lens[pick] > 0]:
        _check(got[o], pts[po[o] : po[o + 1]], 1.5)
