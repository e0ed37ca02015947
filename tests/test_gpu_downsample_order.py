"""Downsampling does not depend on the order in which the points of a voxel reach its list:
voxels of 6 to 40 points whose times cancel (large, middle and small magnitudes and their
negatives), so that whether the partial sums are exact depends on the order in which they
are taken.  The mean is the binary64 sum in index order, rounded to float32, on every
run."""
import numpy as np
import pytest

import oracle
from paper_2202_00242_gb300 import api

from test_gpu_parity import cu, dev  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _voxels(members, voxels, seed):
    """`voxels` voxels of `members` points; in index order the sum of the times loses the
    smallest term's last bit, which a sum of the cancelling pairs first would keep."""
    rng = np.random.default_rng(seed)
    small = np.float32(2.0 ** -20) * (1 + rng.integers(1, 1 << 23, voxels) * 2.0 ** -23)
    mid = 1 + (2 * rng.integers(0, 1 << 22, voxels) + 1) * 2.0 ** -23
    t = np.zeros((members, voxels))
    t[0], t[1], t[2], t[3], t[4] = 2.0 ** 30, small, mid, -2.0 ** 30, -mid
    x = np.arange(voxels) % 40 + rng.uniform(0.1, 0.9, (members, voxels))
    y = np.arange(voxels) // 40 + rng.uniform(0.1, 0.9, (members, voxels))
    pts = np.stack([x, y, np.full_like(x, 0.5)], -1).reshape(-1, 3).astype(np.float32)
    return pts, t.reshape(-1).astype(np.float32)


@pytest.mark.parametrize("members", [6, 8, 9, 12, 32, 40])
def test_times_that_cancel(dev, members):  # noqa: F811
    pts, t = _voxels(members, 1600, members)
    rp, rt, rc = oracle.downsample(pts, t, 1.0, 0.0)
    assert len(rc) == 1600 and np.all(rc == members)
    for _ in range(5):
        gp, gt, gc, _ = api.downsample(cu(pts), 1.0, times=cu(t), split=0.0)
        assert np.array_equal(gc.cpu().numpy(), rc) and np.array_equal(gp.cpu().numpy(), rp)
        assert np.array_equal(gt.cpu().numpy(), rt)


@pytest.mark.parametrize("members", [2, 4, 8, 10, 16, 48, 128])
@pytest.mark.parametrize("tiny", [0.0, 2.0 ** -40])
def test_means_on_midpoints(dev, members, tiny):  # noqa: F811
    """Coordinates of 24 bits, so that the quotients of lists of even length often fall on the
    midpoint of two float32 values; with one much smaller coordinate and time in each voxel
    the sums need more bits than binary64 has."""
    rng = np.random.default_rng(members)
    voxels = 400
    x = np.arange(voxels) % 20 + 1.0 + np.floor(rng.random((members, voxels)) * 2 ** 19) / 2 ** 19
    y = np.arange(voxels) // 20 + 1.0 + np.floor(rng.random((members, voxels)) * 2 ** 19) / 2 ** 19
    z = np.floor(rng.random((members, voxels)) * 2 ** 24) / 2 ** 24
    t = np.floor(rng.random((members, voxels)) * 2 ** 24) / 2 ** 24
    if tiny:
        z[0], t[1 % members] = tiny, tiny
    order = rng.permutation(members * voxels)
    pts = np.stack([x, y, z], -1).reshape(-1, 3).astype(np.float32)[order]
    t = t.reshape(-1).astype(np.float32)[order]
    rp, rt, rc = oracle.downsample(pts, t, 1.0, 0.0)
    assert np.all(rc == members)
    gp, gt, gc, _ = api.downsample(cu(pts), 1.0, times=cu(t), split=0.0)
    assert np.array_equal(gc.cpu().numpy(), rc) and np.array_equal(gp.cpu().numpy(), rp)
    assert np.array_equal(gt.cpu().numpy(), rt)
