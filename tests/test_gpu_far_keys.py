"""Voxel keys of source points so far out that float32 places them more than 2^22 voxels
from where they are: coordinates of 2^48 to 2^52 voxels, which a rotation and a translation
bring back to the map.  The key is that of binary64, so such a point finds its voxel, in
every kernel: the per-point one (a grid of its own), with and without debug outputs, its
27-neighbour form, and the kernels for few items."""
import numpy as np
import pytest
import torch

from paper_2202_00242_gb300 import api, synth

from test_gpu_parity import cu, dev  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

R = 0.25


def _far(seed):
    """A point, a pose that brings it near the origin, and its binary64 key."""
    rng = np.random.default_rng(seed)
    x = (rng.uniform(0.5, 1.0, 3) * rng.choice([-1, 1], 3) * 2.0 ** rng.integers(48, 53) * R)
    x = x.astype(np.float32)
    T = synth.perturb_pose(rng, np.eye(4), 0.0, 40.0)
    x64 = x.astype(np.float64)
    s = np.array([(T[a, 0] * x64[0] + T[a, 1] * x64[1]) + T[a, 2] * x64[2] for a in range(3)])
    T[:3, 3] = -s + rng.uniform(-1.0, 1.0, 3)
    key = np.floor((s + T[:3, 3]) / R)
    q32 = T[:3, :3].astype(np.float32) @ x + T[:3, 3].astype(np.float32)
    return x, T, key, bool(np.abs(q32 / R).max() >= 2.0 ** 22)


@pytest.mark.parametrize("neighbours", [1, 27])
def test_far_points_find_their_voxels(dev, neighbours):  # noqa: F811
    g = (np.arange(-9, 9) + 0.5) * R  # every voxel within 9 of the origin
    tgt = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3).astype(np.float32)
    iso = np.array([0.02, 0, 0, 0.02, 0, 0.02], np.float32)
    vm = api.VoxelMap.build(cu(tgt), cu(np.tile(iso, (len(tgt), 1))), R)
    vm.status()
    beyond = 0
    for seed in range(40):
        x, T, key, out = _far(seed)
        if np.abs(key).max() > 7:
            continue
        beyond += out
        P, C = cu(np.tile(x, (300, 1))), cu(np.tile(iso, (300, 1)))
        want = 300 * neighbours
        dbg = api.linearize(vm, P, C, T, neighbours=neighbours, corr=True, qkeys=True)
        assert np.array_equal(dbg.qkeys.cpu().numpy(), np.tile(key, (300, 1)).astype(np.int64))
        for kw in ({}, {"grid": 2}, {"tile": 4096}, {"variant": 2}, {"variant": 3}):
            lin = api.linearize(vm, P, C, T, neighbours=neighbours, **kw)
            assert int(lin.inliers) == int(dbg.inliers) == want, (seed, kw)
        assert torch.equal(api.linearize(vm, P, C, T, neighbours=neighbours, grid=2).out, dbg.out)
        if neighbours == 1:
            rate = api.overlap_batched([vm], [(P, C)], [[0, 0]], T[None])
            assert float(rate[0][0]) == 1.0
    assert beyond >= 20
