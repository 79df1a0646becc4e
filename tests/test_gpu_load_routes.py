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
