"""The smallest loads: one or two observations among 1 to 70,001 scans (no to
three digits of scan ids, on both sides of each), in either precision, the
state reset afterwards (which re-anchors from what the load kept).  A sort of a
single element makes no pass, so its result stays where it was put."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mm():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2608_14266_gb300 as mm
    assert torch.cuda.is_available()
    return mm


@pytest.mark.parametrize("n_scans", [1, 2, 256, 257, 65537, 70001])
@pytest.mark.parametrize("n_obs", [1, 2])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_few_observations(mm, n_scans, n_obs, precision):
    """Cost, gradient and Hessian against the oracle at the tolerances of each
    path (1e-10 and 1e-11 in FP64; in mixed precision 1e-4 of a single voxel's
    eigenvalue, which is the cost here, and 1e-5), the gradient, which one
    observation leaves at zero, at those of the Hessian; the bits of the first
    state again after an iteration and a reset."""
    import torch
    rng = np.random.default_rng(n_scans)
    pts = rng.normal(size=(8 * n_obs, 3)) * [1.0, 0.7, 0.02] + np.repeat(rng.normal(size=(n_obs, 3)) * 0.05, 8, axis=0)
    cen = oracle.points_to_centred(np.arange(n_obs + 1, dtype=np.int64) * 8, pts)
    off = np.array([0, n_obs], dtype=np.int64)
    scan = np.minimum(np.arange(n_obs) + n_scans // 2, n_scans - 1).astype(np.int32)
    pose = np.zeros((n_scans, 12))
    pose[:, [0, 4, 8]] = 1.0
    pose[:, 9:] = rng.normal(size=(n_scans, 3)) * 0.05
    prob = oracle.ObsProblem(n_scans, off, scan, cen)
    c_ref, planes = oracle.voxel_pass(prob, pose)
    g_ref, H_ref = oracle.grad_hess(prob, pose, planes)
    mixed = precision == "mixed"
    tol = 1e-5 * np.abs(H_ref).max() if mixed else 1e-11 * np.abs(H_ref).max()
    host = (off, scan, cen, pose)
    for args in (host, tuple(torch.from_numpy(x).cuda() for x in host)):
        with mm.BundleAdjuster(precision=mm.BA_MIXED if mixed else mm.BA_FP64, fixed_scan=-1) as ba:
            ba.load_observations(n_scans, *args)
            assert ba.cost() == pytest.approx(c_ref, rel=1e-4 if mixed else 1e-10)
            first = (ba.cost(), *ba.gradient())
            np.testing.assert_allclose(first[1], g_ref, rtol=0, atol=tol)
            np.testing.assert_allclose(first[2], H_ref, rtol=0, atol=tol)
            ba.iterate(1)
            ba.set_state(pose)
            for a, b in zip(first, (ba.cost(), *ba.gradient())):
                np.testing.assert_array_equal(np.asarray(a), np.asarray(b))
