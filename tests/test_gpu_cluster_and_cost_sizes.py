"""Point clusters and the allocation-free cost where their kernels branch:
observations on both sides of the 126 points that the sums of 32-bit halves
hold, spreads at their bound, blocks of uneven observations; voxels of uneven
length around a block's 64."""
import numpy as np
import pytest

import oracle
import scenegen

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


def _clusters(mm, po, pts):
    import torch
    out = torch.empty((len(po) - 1, 10), dtype=torch.float64, device="cuda")
    mm.ba_aggregate_points(torch.from_numpy(po).cuda(), torch.from_numpy(pts).cuda(), out)
    torch.cuda.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("lens", [[1], [2, 1], [125, 126, 127, 128, 3], "ragged", [126] * 300])
@pytest.mark.parametrize("spread", [0.5, 7.95, 15.9])
def test_clusters_around_the_short_sums_bound(mm, lens, spread):
    """Against sums in extended precision: the integer sums are exact in units
    of half p0's last bit (2^-53 here, coordinates of 1 to 2), so an entry of
    the record is off by the rounding of its points to that unit (n 2 spread
    2^-53), of the conversions and of the final multiply-add (a few eps).  A
    spread of 7.95 is just inside the integers' 2^56 units; 15.9 is past it
    and takes FP64 sums, off by the recursive-summation bound, n eps times
    the sum of the terms' sizes."""
    rng = np.random.default_rng(7)
    if lens == "ragged":
        lens = [int(x) for x in rng.integers(1, 400, 700)]
    po = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    pts = rng.uniform(-spread, spread, (po[-1], 3))
    # the bound of the high halves' and cross products' sums: corners of the cube, alike in sign
    pts[rng.random(po[-1]) < 0.5] = spread
    for o in range(len(lens)):
        p0 = np.array([1.75, 1.0, 1.0 / 3.0])
        pts[po[o]:po[o + 1]] += p0
        pts[po[o]] = p0
    got = _clusters(mm, po, pts)
    np.testing.assert_array_equal(got[:, 9], np.diff(po))
    for o in range(len(lens)):
        x = pts[po[o]:po[o + 1]].astype(np.longdouble)
        n = len(x)
        m = x.mean(0)
        d = x - m
        s = np.array([(d[:, a] * d[:, b]).sum() for a in range(3) for b in range(a, 3)])
        f64 = n * EPS if spread > 8 else 0.0
        assert np.abs(got[o, 6:9] - m).max() <= 2.0**-52 + 4 * EPS * (2 + spread) + f64 * 2 * spread, o
        raw = ((x - x[0]) ** 2).sum()  # size of the sums before the mean is taken off
        assert np.abs(got[o, :6] - s).max() <= n * 2 * spread * 2.0**-52 + (4 * EPS + 2 * f64) * raw, (o, n)


@pytest.mark.parametrize("n_voxels", [1, 63, 64, 65, 129, 700])
def test_cost_without_allocation_over_sizes(mm, n_voxels):
    import torch
    s = scenegen.make_scene(scenegen.SceneParams(n_scans=45, n_voxels=n_voxels, obs_min=1, obs_max=45, pts_per_obs=10,
                                                 noise_sigma=0.02, rot_sigma_deg=0.5, trans_sigma=0.05, seed=n_voxels))
    cen = oracle.points_to_centred(s.point_offsets(), s.points())
    c_ref, planes = oracle.voxel_pass(oracle.ObsProblem(s.n_scans, s.voxel_off, s.obs_scan, cen), s.pose_init)
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    cost = torch.zeros(1, dtype=torch.float64, device="cuda")
    lam = torch.zeros(n_voxels, dtype=torch.float64, device="cuda")
    args = (s.n_scans, T(s.voxel_off), T(s.obs_scan), T(cen), T(s.pose_init), cost, lam)
    for _ in range(2):  # the scratch is used again
        mm.ba_eval_cost_noalloc(*args)
        assert float(cost) == pytest.approx(c_ref, rel=1e-10)
    np.testing.assert_allclose(lam.cpu().numpy(), planes[:, 0], rtol=1e-9, atol=1e-15)
    # a scan id out of range in one voxel's last observation: that voxel is NaN, and the cost
    bad = s.obs_scan.copy()
    bad[s.voxel_off[n_voxels // 2 + 1] - 1] = s.n_scans
    mm.ba_eval_cost_noalloc(s.n_scans, T(s.voxel_off), T(bad), T(cen), T(s.pose_init), cost, lam)
    got = lam.cpu().numpy()
    assert np.isnan(float(cost)) and np.isnan(got[n_voxels // 2])
    keep = np.arange(n_voxels) != n_voxels // 2
    np.testing.assert_allclose(got[keep], planes[keep, 0], rtol=1e-9, atol=1e-15)
