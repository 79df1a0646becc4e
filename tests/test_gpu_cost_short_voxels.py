"""The allocation-free cost gives a voxel to one lane from 25,000 voxels of up to
14 observations on average, to four lanes else: both sides of each line, and
scan ids and offsets that are not valid."""
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


@pytest.mark.parametrize("n_voxels,mean", [(24999, 3), (25000, 1), (25000, 3), (25001, 14), (25003, 15), (60001, 6)])
def test_cost_on_both_sides_of_the_lane_line(mm, n_voxels, mean):
    """Tolerances of the cost without allocation: 1e-10 of the cost, 1e-9 of an
    eigenvalue (and 1e-15)."""
    import torch
    rng = np.random.default_rng(n_voxels + mean)
    lens = np.full(n_voxels, mean)
    shift = rng.integers(0, mean, n_voxels // 2)  # uneven lengths, the mean exactly as given
    lens[: n_voxels // 2] -= shift
    lens[n_voxels // 2 : n_voxels // 2 * 2] += shift
    off = np.concatenate([[0], np.cumsum(rng.permutation(lens))]).astype(np.int64)
    n_obs, n_scans = int(off[-1]), 31
    assert n_obs == mean * n_voxels
    vox = np.repeat(np.arange(n_voxels), np.diff(off))
    scan = rng.integers(0, n_scans, n_obs).astype(np.int32)
    axes = np.linalg.qr(rng.normal(size=(n_voxels, 3, 3)))[0][vox]
    D = np.array([9.0, 4.0, 0.004]) * rng.uniform(0.5, 1.5, (n_obs, 3))
    S = np.einsum("oij,oj,okj->oik", axes, D, axes)
    m = rng.normal(size=(n_voxels, 3))[vox] * 5.0
    m += np.einsum("oij,oj->oi", axes, rng.normal(size=(n_obs, 3)) * [0.5, 0.5, 0.01])
    agg = np.concatenate([S[:, [0, 0, 0, 1, 1, 2], [0, 1, 2, 1, 2, 2]], m, np.full((n_obs, 1), 10.0)], 1)
    pose = np.zeros((n_scans, 12))
    pose[:, [0, 4, 8]] = 1.0
    pose[:, 9:] = rng.normal(size=(n_scans, 3)) * 0.01
    c_ref, planes = oracle.voxel_pass(oracle.ObsProblem(n_scans, off, scan, agg), pose)
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    cost = torch.zeros(1, dtype=torch.float64, device="cuda")
    lam = torch.zeros(n_voxels, dtype=torch.float64, device="cuda")
    first = None
    for _ in range(3):  # the scratch is used again; the same bits
        mm.ba_eval_cost_noalloc(n_scans, T(off), T(scan), T(agg), T(pose), cost, lam)
        first = float(cost) if first is None else first
        assert float(cost) == first == pytest.approx(c_ref, rel=1e-10)
    np.testing.assert_allclose(lam.cpu().numpy(), planes[:, 0], rtol=1e-9, atol=1e-15)
    # a scan id out of range in one voxel, an empty voxel: those are NaN, and the cost
    bad_scan, bad_off = scan.copy(), off.copy()
    hit = n_voxels - 7
    bad_scan[off[hit + 1] - 1] = n_scans
    bad_off[101] = bad_off[100]
    mm.ba_eval_cost_noalloc(n_scans, T(bad_off), T(bad_scan), T(agg), T(pose), cost, lam)
    got = lam.cpu().numpy()
    assert np.isnan(float(cost)) and np.isnan(got[hit]) and np.isnan(got[100])
    keep = np.ones(n_voxels, bool)
    keep[[hit, 100, 101]] = False  # (101 has the observations of 100 as well)
    np.testing.assert_allclose(got[keep], planes[keep, 0], rtol=1e-9, atol=1e-15)
