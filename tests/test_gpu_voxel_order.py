"""Order of the voxel-grouped cloud: voxels of a map by Morton code of the low 10
key bits per axis (x lowest), ties by voxel id, in chunks of 16,384 voxel ids; points
of a voxel by index.  At the edges of the radix sort: one voxel, one element per lane
and one more, a full chunk, two chunks, keys within one voxel of the origin, across
the sign, and wide enough to use (and to wrap) all 10 bits."""
import numpy as np
import pytest

from paper_2202_00242_gb300 import api

from test_gpu_parity import cu, dev  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _spread(v):
    out = np.zeros_like(v)
    for b in range(10):
        out |= ((v >> b) & 1) << (3 * b)
    return out


def _expected(points, r):
    k = np.floor(points.astype(np.float64) / r).astype(np.int64)
    _, first, inv = np.unique(k, axis=0, return_index=True, return_inverse=True)
    vid = np.argsort(np.argsort(first))[inv.ravel()]          # order of first appearance
    m = k & 1023
    code = _spread(m[:, 0]) | (_spread(m[:, 1]) << 1) | (_spread(m[:, 2]) << 2)
    return np.lexsort((np.arange(len(points)), vid, code, vid // 16384))


@pytest.mark.parametrize("n,extent", [
    (1, 0.4), (40, 0.4), (31, 3.0), (33, 60.0), (1024, 60.0), (1025, 60.0), (5000, 0.9),
    (5000, 30.0), (16384, 200.0), (20000, 500.0), (40000, 2000.0), (70000, 45.0)])
def test_grouped_order(dev, n, extent):  # noqa: F811
    rng = np.random.default_rng(n)
    pts = rng.uniform(-extent, extent, (n, 3)).astype(np.float32)
    covs = rng.uniform(0.5, 1.0, (n, 6)).astype(np.float32)
    order = _expected(pts, 1.0)
    vm = api.VoxelMap.build(cu(pts), cu(covs), 1.0)
    for again in range(2):
        if again:
            api.rebuild_voxelmaps([vm], cu(pts), cu(covs))
        vm.status()
        gp, gc = vm.grouped_cloud()
        assert np.array_equal(gp.cpu().numpy(), pts[order])
        assert np.array_equal(gc.cpu().numpy(), covs[order])
