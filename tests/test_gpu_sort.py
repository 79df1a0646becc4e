"""The library's radix sort through the paths that use it, at sizes around a
tile (4,096) and with keys that leave one digit's run in every tile: the
layout of a load (voxel order, scan-major order) and the preprocessing's order,
both of which must be exactly those of a stable sort."""
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


@pytest.mark.parametrize("n", [1, 2, 4095, 4096, 4097, 8192, 12289, 700001])
@pytest.mark.parametrize("cells", [1, 3, 300, 70000])
def test_preprocessing_order_is_a_stable_sort(mm, n, cells):
    """Points on a line of `cells` voxels in random order, three scans: voxels
    ascending, scans ascending inside, counts per (voxel, scan).  One cell: every
    key equal; 70,000: three digits."""
    rng = np.random.default_rng(n + cells)
    cell = rng.integers(0, cells, n)
    P = np.zeros((n, 3))
    P[:, 0] = cell + 0.5
    cut = sorted(int(x) for x in rng.integers(0, n + 1, 2))
    spo = np.array([0, *cut, n], dtype=np.int64)
    scan = np.repeat(np.arange(3), np.diff(spo))
    poses = np.tile(np.concatenate([np.eye(3).ravel(), np.zeros(3)]), (3, 1))
    got = mm.voxelize(spo, P, poses, 1.0)
    pairs, counts = np.unique(cell * 3 + scan, return_counts=True)
    np.testing.assert_array_equal(got["obs_scan"], pairs % 3)
    np.testing.assert_array_equal(got["agg"][:, 9], counts)
    voxels, first = np.unique(pairs // 3, return_index=True)
    np.testing.assert_array_equal(got["index"][:, 0], voxels)
    np.testing.assert_array_equal(got["voxel_off"][:-1], first)


@pytest.mark.parametrize("n_scans,n_voxels", [(2, 1), (3, 4096), (300, 4097), (70000, 9000)])
def test_loaded_layout_gives_the_oracle_gradient(mm, n_scans, n_voxels):
    """One to three digits of scan ids, voxel counts around a tile: a misplaced
    observation would change its scan's gradient (tolerance of the FP64 path's
    element comparisons)."""
    rng = np.random.default_rng(n_voxels)
    lens = rng.integers(1, 4, n_voxels)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    scan = rng.integers(0, n_scans, off[-1]).astype(np.int32)
    A = rng.normal(size=(off[-1], 3, 3)) * 0.1
    S = A @ A.transpose(0, 2, 1)
    agg = np.concatenate([S[:, [0, 0, 0, 1, 1, 2], [0, 1, 2, 1, 2, 2]], rng.normal(size=(off[-1], 3)),
                          np.full((off[-1], 1), 9.0)], 1)
    poses = np.tile(np.concatenate([np.eye(3).ravel(), np.zeros(3)]), (n_scans, 1))
    poses[:, 9:] = rng.normal(size=(n_scans, 3))
    prob = oracle.ObsProblem(n_scans, off, scan, agg)
    c, planes = oracle.voxel_pass(prob, poses)
    g, H = oracle.grad_hess(prob, poses, planes)
    with mm.BundleAdjuster() as ba:
        ba.load_observations(n_scans, off, scan, agg, poses)
        assert ba.cost() == pytest.approx(c, rel=1e-10)
        g2, H2 = ba.gradient()
    # (a voxel seen by one scan has no gradient: what is left of it is the
    # rounding of terms of the Hessian's size)
    np.testing.assert_allclose(g2, g, rtol=0, atol=1e-10 * np.abs(g).max() + 1e-13 * np.abs(H).max())
    np.testing.assert_allclose(H2, H, rtol=0, atol=1e-11 * np.abs(H).max())


@pytest.mark.parametrize("n", [4096 * 4096 - 1, 4096 * 4096 + 5])
def test_prefix_sums_on_both_sides_of_4096_tiles(mm, n):
    """A point to a voxel, so that the prefix sums run over n + 1 heads: up to
    4,096 tiles of 4,096 a block adds up the sums of the tiles before its own,
    beyond they are scanned first.  Every voxel starts where it must."""
    import torch
    i = torch.arange(n, dtype=torch.int64, device="cuda")
    cell = torch.stack([i % 300, (i // 300) % 300, i // 90000], 1)
    spo = torch.tensor([0, n], dtype=torch.int64, device="cuda")
    poses = torch.tensor([[1.0, 0, 0, 0, 1, 0, 0, 0, 1, 0, 0, 0]], dtype=torch.float64, device="cuda")
    got = mm.voxelize(spo, cell.double() + 0.5, poses, 1.0, out="device")
    assert torch.equal(got["voxel_off"], torch.arange(n + 1, device="cuda"))
    key = lambda x: (x[:, 0].long() * 300 + x[:, 1].long()) * 300 + x[:, 2].long()
    assert torch.equal(key(got["index"]), key(cell).sort()[0])
