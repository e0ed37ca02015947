"""Rebuilds empty the previous build's lookup slots inside the insertion, whose errors
reach the status through the numbering: at sizes of one block, of eight and nine blocks,
and on both numbering paths (32 x 32,768 points and more), a rebuild equals a fresh build
(no slot of the previous one is found), an error is reported, and the next rebuild is
sound again."""
import numpy as np
import pytest
import torch

from paper_2202_00242_gb300 import api
from paper_2202_00242_gb300._lib import VGICPError

from test_gpu_parity import cu, dev  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 256, 2048, 2049, 2305, 20000, 32 * 32768 + 40])
def test_rebuild_after_an_error(dev, n):  # noqa: F811
    rng = np.random.default_rng(n)
    a = rng.uniform(-20, 20, (n, 3)).astype(np.float32)
    b = (a * np.float32(0.25) + np.float32(3.0)).astype(np.float32)
    covs = cu(np.tile(np.array([1, 0, 0, 1, 0, 1], np.float32), (n, 1)))
    bad = b.copy()
    bad[n // 2, 1] = np.float32(3.0e7)
    src = cu(np.concatenate([a, b])), cu(np.tile(np.array([1, 0, 0, 1, 0, 1], np.float32), (2 * n, 1)))
    T = np.eye(4)
    fresh = {}
    for k, p in (("a", a), ("b", b)):
        vm = api.VoxelMap.build(cu(p), covs, 1.0)
        fresh[k] = (vm.export(), api.linearize(vm, *src, T))
    vm = api.VoxelMap.build(cu(a), covs, 1.0)
    for k, p in (("b", b), ("a", a), (None, bad), (None, bad), ("b", b), ("a", a)):
        api.rebuild_voxelmaps([vm], cu(p), covs)
        if k is None:
            with pytest.raises(VGICPError) as e:
                vm.status()
            assert e.value.code == -4
            continue
        vm.status()
        ex, lin = vm.export(), api.linearize(vm, *src, T)
        want, ref = fresh[k]
        for f in want:
            assert np.array_equal(ex[f], want[f])
        assert torch.equal(lin.out, ref.out) and torch.equal(lin.inliers, ref.inliers)
