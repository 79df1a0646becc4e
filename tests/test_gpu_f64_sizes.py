"""The FP64 passes over problem sizes: the voxel pass gives 8, 16 or 32 voxels
to a block by the number of voxels, so sizes on both sides of each line, one
voxel, and ragged last blocks; the scan pass's reduction and rotation with
scans of one observation up to several hundred."""
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


@pytest.mark.parametrize("n_voxels", [1, 7, 33, 2432, 2433, 6144, 6145])
@pytest.mark.parametrize("gn", [False, True])
def test_fp64_passes_match_oracle_over_sizes(mm, n_voxels, gn):
    """Tolerances: the FP64 path's cost budget (1e-10) and those of the element
    comparisons of g and H (1e-10 and 1e-11 of the largest entry)."""
    s = scenegen.make_scene(scenegen.SceneParams(n_scans=37, n_voxels=n_voxels, obs_min=1, obs_max=35, pts_per_obs=12,
                                                 side_min=0.5, side_max=2.0, noise_sigma=0.02, rot_sigma_deg=0.5,
                                                 trans_sigma=0.05, seed=n_voxels))
    cen = oracle.points_to_centred(s.point_offsets(), s.points())
    prob = oracle.ObsProblem(s.n_scans, s.voxel_off, s.obs_scan, cen)
    c_ref, planes = oracle.voxel_pass(prob, s.pose_init)
    g_ref, H_ref = oracle.grad_hess(prob, s.pose_init, planes, gauss_newton=gn)
    with mm.BundleAdjuster(hessian_mode=int(gn)) as ba:
        ba.load_observations(s.n_scans, s.voxel_off, s.obs_scan, cen, s.pose_init)
        got = ba.planes()
        assert ba.cost() == pytest.approx(c_ref, rel=1e-10)
        np.testing.assert_allclose(got[:, 0], planes[:, 0], rtol=1e-9, atol=1e-15)
        np.testing.assert_allclose(got[:, 6:9], planes[:, 6:9], rtol=0, atol=1e-10)
        g, H = ba.gradient()
        np.testing.assert_allclose(g, g_ref, rtol=0, atol=1e-10 * np.abs(g_ref).max())
        for j in range(s.n_scans):
            np.testing.assert_allclose(H[j], H_ref[j], rtol=0, atol=1e-11 * max(np.abs(H_ref[j]).max(), 1e-300))
        st = ba.iterate(2)
    lm = oracle.LM(prob, s.pose_init, gauss_newton=gn)
    for _ in range(2):
        lm.step()
    assert st["cost"] == pytest.approx(lm.cost, rel=1e-9)
