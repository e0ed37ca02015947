"""Voxel statistics and grouped order where the lists per voxel are long: averages on
both sides of each threads-per-voxel step, lists longer than a warp sums alone, one
list over the staging buffer, and covariance entries of very different magnitude
(inexact partial sums).  Everything must equal the oracle's map bit for bit."""
import numpy as np
import pytest

from paper_2202_00242_gb300 import api

from test_gpu_grouped_cloud import check_export, check_grouped
from test_gpu_parity import cu, dev  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _cloud(n, voxels, seed):
    """n points over `voxels` unit voxels, one of them with a tenth of all points."""
    rng = np.random.default_rng(seed)
    v = np.where(rng.random(n) < 0.1, 0, rng.integers(0, voxels, n))
    base = np.column_stack([v % 7, v // 7 % 7, v // 49]) - 3
    pts = (base + rng.uniform(0.01, 0.99, (n, 3))).astype(np.float32)
    covs = rng.uniform(0.5, 1.0, (n, 6)).astype(np.float32)
    covs[:, [1, 2, 4]] *= np.float32(10.0) ** rng.integers(-7, 0, (n, 3)).astype(np.float32)
    return pts, covs


@pytest.mark.parametrize("n,voxels", [(1, 1), (130, 11), (700, 64), (1100, 34), (2600, 33),
                                      (5000, 41), (6000, 12), (9000, 9), (40000, 100),
                                      (30000, 3)])
def test_long_lists(dev, n, voxels):  # noqa: F811
    pts, covs = _cloud(n, voxels, n + voxels)
    vm = api.VoxelMap.build(cu(pts), cu(covs), 1.0)
    vm.status()
    check_export(vm, pts, covs, 1.0)
    check_grouped(vm, pts, covs, 1.0)


def test_rebuild_from_short_to_long_lists(dev):  # noqa: F811
    """The kernel is picked by the first build; a rebuild may look different."""
    short, cs = _cloud(6000, 330, 1)
    short *= np.float32(9.0)
    long, cl = _cloud(6000, 20, 2)
    for first, second in (((short, cs), (long, cl)), ((long, cl), (short, cs))):
        vm = api.VoxelMap.build(cu(first[0]), cu(first[1]), 1.0)
        api.rebuild_voxelmaps([vm], cu(second[0]), cu(second[1]))
        vm.status()
        check_export(vm, second[0], second[1], 1.0)
        check_grouped(vm, second[0], second[1], 1.0)
