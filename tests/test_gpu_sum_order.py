"""Voxel covariances whose entries cancel (large, middle and small magnitudes and their
negatives, off the diagonal of positive semi-definite matrices), in lists that several
threads or a whole warp sum: the sums are those in ascending point index, and not those of
the threads' shares, which may be exact where that order rounds.  Every voxel equals the
oracle's bit for bit; lists whose quotients fall on midpoints of float32 values do too."""
import numpy as np
import pytest

from paper_2202_00242_gb300 import api

from test_gpu_grouped_cloud import check_export
from test_gpu_parity import cu, dev  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _voxels(members, voxels, seed):
    rng = np.random.default_rng(seed)
    v = np.repeat(np.arange(voxels), members)
    base = np.column_stack([v % 20, v // 20 % 20, v // 400])
    pts = (base + rng.uniform(0.01, 0.99, (len(v), 3))).astype(np.float32)
    return pts, v, rng


@pytest.mark.parametrize("apart,members", [
    (a, m) for a in (1, 2, 4, 8, 16, 32) for m in (8, 12, 24, 40, 70, 200, 2100) if 2 * a + 3 <= m])
def test_entries_that_cancel(dev, members, apart):  # noqa: F811
    voxels = 40 if members > 1000 else 400
    pts, v, rng = _voxels(members, voxels, members + apart)
    off = np.zeros((voxels, members, 3))
    small = 2.0 ** -20 * (1 + rng.integers(1, 1 << 23, (voxels, 3)) * 2.0 ** -23)
    mid = 1 + (2 * rng.integers(0, 1 << 22, (voxels, 3)) + 1) * 2.0 ** -23
    # in index order the small entry is added between the others; `apart` entries on, the
    # large and the middle one are taken back
    off[:, 0], off[:, 1], off[:, 2] = 2.0 ** 30, small, mid
    off[:, 0 + apart if apart > 2 else 3] = -2.0 ** 30
    off[:, 2 + apart if apart > 2 else 4] = -mid
    off = off.reshape(-1, 3)
    diag = np.abs(off).sum(axis=1) + 1.0
    covs = np.column_stack([diag, off[:, 0], off[:, 1], diag, off[:, 2], diag]).astype(np.float32)
    vm = api.VoxelMap.build(cu(pts), cu(covs), 1.0)
    vm.status()
    check_export(vm, pts, covs, 1.0)


@pytest.mark.parametrize("members", [8, 10, 16, 32, 96, 128, 256])
@pytest.mark.parametrize("tiny", [0.0, 2.0 ** -40])
def test_means_on_midpoints(dev, members, tiny):  # noqa: F811
    pts, v, rng = _voxels(members, 200, members)
    pts = (np.floor(pts) + np.floor(rng.random(pts.shape) * 2 ** 18) / 2 ** 18).astype(np.float32)
    covs = (np.floor(rng.random((len(pts), 6)) * 2 ** 24) / 2 ** 24).astype(np.float32)
    covs[:, [0, 3, 5]] += 3.0
    if tiny:
        covs[::members, 1] = tiny
        pts[1::members, 0] = np.where(v[1::members] % 20 == 0, tiny, pts[1::members, 0])
    order = rng.permutation(len(pts))
    pts, covs = pts[order], covs[order]
    vm = api.VoxelMap.build(cu(pts), cu(covs), 1.0)
    vm.status()
    check_export(vm, pts, covs, 1.0)


@pytest.mark.parametrize("members", [8, 24, 70, 200, 2100])
@pytest.mark.parametrize("scale", [1e-6, 1e-9, 1e-20, 0.0])
def test_entries_that_are_all_tiny(dev, members, scale):  # noqa: F811
    """Planes along an axis: off-diagonal entries far below the diagonal ones, in one list in
    three with a larger one among them."""
    pts, v, rng = _voxels(members, 40 if members > 1000 else 300, members)
    off = rng.normal(size=(len(v), 3)) * scale
    off[::3 * members, 1] = 0.25
    covs = np.column_stack([1 + rng.random(len(v)), off[:, 0], off[:, 1], 1 + rng.random(len(v)),
                            off[:, 2], np.full(len(v), 1.0)]).astype(np.float32)
    vm = api.VoxelMap.build(cu(pts), cu(covs), 1.0)
    vm.status()
    check_export(vm, pts, covs, 1.0)
