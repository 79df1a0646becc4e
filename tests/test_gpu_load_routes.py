"""Where a load's kernels branch: clusters in device memory at 16-byte and
8-byte alignment (paired or single values), host clusters in one copy or in
chunks, both cluster forms, voxels of one observation up to more than a
window's slices; and a reset of the state after each kind of load, which
re-anchors from what the load kept."""
import numpy as np
import pytest

import oracle
import scenegen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mm():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2608_14266_gb300 as mm
    assert torch.cuda.is_available()
    return mm


def _device(a, shift):
    """a on the device, starting `shift` doubles behind an allocation's start."""
    import torch
    t = torch.empty(a.size + shift, dtype=torch.float64, device="cuda")
    t[shift:] = torch.from_numpy(np.ascontiguousarray(a).reshape(-1)).cuda()
    return t[shift:].view(a.shape)


@pytest.mark.parametrize("n_voxels", [1, 31, 700, 70000])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_load_routes_agree(mm, n_voxels, precision):
    """The route decides how the clusters are read, never a value: every route
    gives the same cost, gradient and poses bit for bit."""
    import torch
    s = scenegen.make_scene(scenegen.SceneParams(n_scans=37, n_voxels=n_voxels, obs_min=1, obs_max=9, pts_per_obs=6,
                                                 side_min=0.5, side_max=2.0, noise_sigma=0.02, rot_sigma_deg=0.5,
                                                 trans_sigma=0.05, seed=n_voxels))
    cen = oracle.points_to_centred(s.point_offsets(), s.points())
    off, scan = np.asarray(s.voxel_off, np.int64), np.asarray(s.obs_scan, np.int32)
    pose = np.asarray(s.pose_init, np.float64)
    prec = mm.BA_MIXED if precision == "mixed" else mm.BA_FP64

    def run(load):
        with mm.BundleAdjuster(precision=prec) as ba:
            load(ba)
            first = (ba.cost(), *ba.gradient())
            ba.iterate(3)
            poses = ba.poses().copy()
            ba.set_state(pose)
            again = (ba.cost(), *ba.gradient())
            return first, poses, again

    dev = lambda shift: (lambda ba: ba.load_observations(
        s.n_scans, torch.from_numpy(off).cuda(), torch.from_numpy(scan).cuda(), _device(cen, shift),
        torch.from_numpy(pose).cuda()))
    host = lambda ba: ba.load_observations(s.n_scans, off, scan, cen, pose)
    want = run(dev(0))
    for load in (dev(1), host):
        got = run(load)
        for a, b in zip(want[0] + (want[1],) + want[2], got[0] + (got[1],) + got[2]):
            np.testing.assert_array_equal(np.asarray(a), np.asarray(b))
    for a, b in zip(want[0], want[2]):
        np.testing.assert_array_equal(np.asarray(a), np.asarray(b))


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("row,col", [(0, 0), (511, 9), (2047, 5), (-1, 9)])
def test_bad_cluster_is_named(mm, shift, row, col):
    """A value that is not finite, or a count below one, in any column of any
    row is refused with that row."""
    import torch
    s = scenegen.make_scene(scenegen.SceneParams(n_scans=37, n_voxels=700, obs_min=2, obs_max=9, pts_per_obs=6,
                                                 side_min=0.5, side_max=2.0, noise_sigma=0.02, rot_sigma_deg=0.5,
                                                 trans_sigma=0.05, seed=4))
    cen = oracle.points_to_centred(s.point_offsets(), s.points()).copy()
    cen[row, col] = 0.0 if col == 9 else np.inf
    row = row % len(cen)
    args = (torch.from_numpy(np.asarray(s.voxel_off, np.int64)).cuda(),
            torch.from_numpy(np.asarray(s.obs_scan, np.int32)).cuda(), _device(cen, shift),
            torch.from_numpy(np.asarray(s.pose_init, np.float64)).cuda())
    for prec in (mm.BA_MIXED, mm.BA_FP64):
        with mm.BundleAdjuster(precision=prec) as ba:
            with pytest.raises(Exception, match=rf"\b{row}\b"):
                ba.load_observations(s.n_scans, *args)


@pytest.mark.parametrize("n_scans", [1, 1024, 1025, 70001])
@pytest.mark.parametrize("long_voxel", [0, 6000])
def test_scan_order_and_slot_bound(mm, n_scans, long_voxel):
    """The block order of the scans (ranked in one block up to 1024 scans, else
    sorted) names every scan once, those without an observation included; the
    number of slots is taken from its bound, or, with one voxel far longer than
    the others, read back.  Compared with the oracle at the FP64 path's
    tolerances (1e-10 of the largest entry of g, 1e-11 of H's; with one scan g
    is zero, a sum that cancels, and is compared at H's)."""
    rng = np.random.default_rng(n_scans)
    lens = rng.integers(1, 12, 900)
    if long_voxel:
        lens[450] = long_voxel
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    n_obs = int(off[-1])
    # half of the observations on few scans, so that lengths differ and tie
    scan = np.where(rng.random(n_obs) < 0.5, rng.integers(0, max(n_scans // 50, 1), n_obs),
                    rng.integers(0, n_scans, n_obs)).astype(np.int32)
    pts = rng.normal(size=(n_obs, 8, 3)) * [1.0, 0.7, 0.02] + rng.normal(size=(n_obs, 1, 3))
    cen = oracle.points_to_centred(np.arange(n_obs + 1, dtype=np.int64) * 8, pts.reshape(-1, 3))
    pose = np.zeros((n_scans, 12))
    pose[:, [0, 4, 8]] = 1.0
    pose[:, 9:] = rng.normal(size=(n_scans, 3))
    prob = oracle.ObsProblem(n_scans, off, scan, cen)
    c_ref, planes = oracle.voxel_pass(prob, pose)
    g_ref, H_ref = oracle.grad_hess(prob, pose, planes, gauss_newton=False)
    with mm.BundleAdjuster() as ba:
        ba.load_observations(n_scans, off, scan, cen, pose)
        assert ba.cost() == pytest.approx(c_ref, rel=1e-10)
        g, H = ba.gradient()
        g_tol = 1e-10 * np.abs(g_ref).max() if n_scans > 1 else 1e-11 * np.abs(H_ref).max()
        np.testing.assert_allclose(g, g_ref, rtol=0, atol=g_tol)
        np.testing.assert_allclose(H, H_ref, rtol=0, atol=1e-11 * np.abs(H_ref).max())
