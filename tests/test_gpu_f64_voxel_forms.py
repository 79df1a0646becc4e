"""The FP64 voxel pass has one thread, or 4, 8 or 16, to a voxel by a problem's
voxels and observations, and a batch that fills the GPU runs all of these with a
thread to a voxel: jobs on both sides of each line give the bits they have alone
in a small and in a large batch, and the form for many short voxels the
oracle's planes."""
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


def _problem(n_voxels, lo, hi, n_scans=23):
    """Planar voxels seen from poses near the identity, lo..hi observations each."""
    rng = np.random.default_rng(n_voxels + hi)
    lens = rng.integers(lo, hi + 1, n_voxels)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    n_obs = int(off[-1])
    vox = np.repeat(np.arange(n_voxels), lens)
    scan = ((vox + np.arange(n_obs) * 7) % n_scans).astype(np.int32)
    axes = np.linalg.qr(rng.normal(size=(n_voxels, 3, 3)))[0][vox]
    D = np.array([9.0, 4.0, 0.004]) * rng.uniform(0.5, 1.5, (n_obs, 3))
    S = np.einsum("oij,oj,okj->oik", axes, D, axes)
    centre = rng.normal(size=(n_voxels, 3)) * 5.0
    mean = centre[vox] + np.einsum("oij,oj->oi", axes, rng.normal(size=(n_obs, 3)) * [0.5, 0.5, 0.01])
    agg = np.concatenate([S[:, [0, 0, 0, 1, 1, 2], [0, 1, 2, 1, 2, 2]], mean, np.full((n_obs, 1), 10.0)], 1)
    pose = np.zeros((n_scans, 12))
    pose[:, [0, 4, 8]] = 1.0
    pose[:, 9:] = rng.normal(size=(n_scans, 3)) * 0.01
    return n_scans, off, scan, agg, pose


JOBS = [(1, 3, 3), (100, 1, 35), (2432, 1, 20), (2433, 1, 20), (6144, 1, 9), (6145, 1, 9), (7000, 20, 40)]
MANY = [(49999, 1, 3), (50000, 1, 3), (50001, 1, 15), (50007, 9, 14)]


def test_batches_give_the_bits_of_jobs_alone(mm):
    jobs = [_problem(*j) for j in JOBS + MANY]
    alone = []
    for ns, off, scan, agg, pose in jobs:
        with mm.BundleAdjuster() as ba:
            ba.load_observations(ns, off, scan, agg, pose)
            st = ba.iterate(3)
            alone.append((ba.poses().copy(), st["cost"], st["mu"], ba.planes()))
    # 24,255 voxels (below a large batch's 50,000), with those of 50,000 each, and
    # two of the latter by themselves
    for pick in (range(len(JOBS)), range(len(jobs)), [len(JOBS)], [len(JOBS) + 1]):
        bas = [mm.BundleAdjuster() for _ in pick]
        with mm.Batch() as b:
            for ba, k in zip(bas, pick):
                ns, off, scan, agg, pose = jobs[k]
                ba.load_observations(ns, off, scan, agg, pose)
                b.add(ba)
            b.iterate(3)
            for ba, k in zip(bas, pick):
                poses, cost, mu, planes = alone[k]
                st = ba.stats()
                np.testing.assert_array_equal(ba.poses(), poses, err_msg=str(k))
                assert (st["cost"], st["mu"]) == (cost, mu), k
                np.testing.assert_array_equal(ba.planes(), planes, err_msg=str(k))
        for ba in bas:
            ba.close()


@pytest.mark.parametrize("job", MANY)
def test_many_short_voxels_match_oracle(mm, job):
    """At the tolerances of the FP64 passes over sizes (1e-10 of the cost, 1e-9 of
    an eigenvalue, 1e-10 of the centroids' metres and of the gradient's largest
    entry)."""
    ns, off, scan, agg, pose = _problem(*job)
    prob = oracle.ObsProblem(ns, off, scan, agg)
    c_ref, planes = oracle.voxel_pass(prob, pose)
    g_ref, H_ref = oracle.grad_hess(prob, pose, planes)
    with mm.BundleAdjuster() as ba:
        ba.load_observations(ns, off, scan, agg, pose)
        got = ba.planes()
        assert ba.cost() == pytest.approx(c_ref, rel=1e-10)
        np.testing.assert_allclose(got[:, 0], planes[:, 0], rtol=1e-9, atol=1e-15)
        np.testing.assert_allclose(got[:, 6:9], planes[:, 6:9], rtol=0, atol=1e-10)
        g, H = ba.gradient()
        np.testing.assert_allclose(g, g_ref, rtol=0, atol=1e-10 * np.abs(g_ref).max())
        np.testing.assert_allclose(H, H_ref, rtol=0, atol=1e-11 * np.abs(H_ref).max())
