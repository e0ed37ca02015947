"""Voxel numbering, table masks and list offsets around the sizes at which their kernels
change: whole and partial words of the first-point bitmap, the most points one CTA
numbers (32 x 32,768) and one more, maps of one and of several sorting chunks beside
empty maps, and rebuilds whose maps change size.  Exported maps and grouped clouds
must equal the definition (numpy) exactly."""
import numpy as np
import pytest

from paper_2202_00242_gb300 import api

from test_gpu_parity import cu, dev  # noqa: F401  (fixture)
from test_gpu_voxel_order import _expected

pytestmark = pytest.mark.gpu


def _cloud(n, extent, seed):
    rng = np.random.default_rng(seed)
    return (rng.uniform(-extent, extent, (n, 3)).astype(np.float32),
            rng.uniform(0.5, 1.0, (n, 6)).astype(np.float32))


def _check(vm, pts, covs):
    if len(pts) == 0:
        assert vm.num_voxels == 0
        return
    k = np.floor(pts.astype(np.float64)).astype(np.int64)
    u, first, cnt = np.unique(k, axis=0, return_index=True, return_counts=True)
    o = np.argsort(first)
    ex = vm.export()
    assert np.array_equal(ex["keys"], u[o]) and np.array_equal(ex["counts"], cnt[o])
    order = _expected(pts, 1.0)
    gp, gc = vm.grouped_cloud()
    assert np.array_equal(gp.cpu().numpy(), pts[order])
    assert np.array_equal(gc.cpu().numpy(), covs[order])


@pytest.mark.parametrize("sizes,extent", [
    ([31], 4.0), ([32], 4.0), ([33, 31, 64], 4.0), ([0, 5, 0, 70, 0], 6.0),
    ([20000, 45000, 3, 17000], 60.0), ([32 * 32768 - 40, 39], 30.0), ([32 * 32768 - 40, 41], 30.0)])
def test_batches(dev, sizes, extent):  # noqa: F811
    clouds = [_cloud(n, extent, 10 + i) for i, n in enumerate(sizes)]
    other = [_cloud(n, extent * 0.4, 50 + i) for i, n in enumerate(sizes)]
    off = np.concatenate([[0], np.cumsum(sizes)])
    cat = lambda cs, j: cu(np.concatenate([c[j] for c in cs]))  # noqa: E731
    maps = api.build_voxelmaps(cat(clouds, 0), cat(clouds, 1), off, 1.0)
    for step in (clouds, other, clouds):
        api.rebuild_voxelmaps(maps, cat(step, 0), cat(step, 1))
        maps[0].status()
        for m, c in zip(maps, step):
            _check(m, *c)
