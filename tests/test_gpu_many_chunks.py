"""Maps of several chunks of 16,384 voxels, in one batch with small and empty ones: each
chunk's point lists start behind those of its map's earlier chunks, whether those are
counted by a kernel of their own (the first build's largest map has more than eight chunks)
or not; rebuilds with many more or fewer voxels than the first build."""
import numpy as np
import pytest

from paper_2202_00242_gb300 import api

from test_gpu_grouped_cloud import check_export
from test_gpu_parity import cu, dev  # noqa: F401  (fixture)
from test_gpu_voxel_order import _expected

pytestmark = pytest.mark.gpu


def _check(maps, pts, covs, off):
    for m, vm in enumerate(maps):
        p, c = pts[off[m]:off[m + 1]], covs[off[m]:off[m + 1]]
        if not len(p):
            continue
        order = _expected(p, 1.0)
        gp, gc = vm.grouped_cloud()
        assert np.array_equal(gp.cpu().numpy(), p[order])
        assert np.array_equal(gc.cpu().numpy(), c[order])
        check_export(vm, p, c, 1.0)


@pytest.mark.parametrize("sizes", [[200000], [3, 60000, 0, 150000, 20000, 32769], [135000, 131072]])
def test_offsets_of_later_chunks(dev, sizes):  # noqa: F811
    rng = np.random.default_rng(len(sizes))
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n = int(off[-1])
    covs = rng.uniform(0.5, 1.0, (n, 6)).astype(np.float32)
    wide = rng.uniform(-300.0, 300.0, (n, 3)).astype(np.float32)   # nearly a voxel a point
    wide[::70] = wide[0]                                           # and one of many points
    mid = rng.uniform(-22.0, 22.0, (n, 3)).astype(np.float32)      # lists of different lengths
    near = rng.uniform(-9.0, 9.0, (n, 3)).astype(np.float32)       # one chunk a map
    for first, later in ((wide, (mid, near, wide)), (near, (wide, mid))):
        maps = api.build_voxelmaps(cu(first), cu(covs), off, 1.0)
        maps[0].status()
        _check(maps, first, covs, off)
        for p in later:
            api.rebuild_voxelmaps(maps, cu(p), cu(covs))
            maps[0].status()
            _check(maps, p, covs, off)
