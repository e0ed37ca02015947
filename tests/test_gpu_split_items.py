"""Few long work items go to the cluster-per-item kernel; any grid request keeps the
per-point kernel.  Both add the same float32 terms in the same order, so H, b, err,
the gradients and the counts must be equal bit for bit, at ragged sizes (tails of
warps, of rounds of 16 points, of items) and on both sides of the item limit."""
import numpy as np
import pytest
import torch

from paper_2202_00242_gb300 import api, synth

from test_gpu_parity import cu, dev  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _plans(sizes, tile, seed=3):
    w = synth.with_surface_covariances(
        synth.outdoor_submaps(seed=seed, n_submaps=len(sizes), n_min=max(sizes), n_max=max(sizes),
                              neighbours=1))
    clouds = [w.clouds.cloud(c) for c in range(len(sizes))]
    maps = [api.VoxelMap.build(cu(p), cu(c), 1.0) for p, c in clouds]
    src = [(cu(p[:n]), cu(c[:n])) for (p, c), n in zip(clouds, sizes)]
    pairs = w.pairs
    return [api.Plan(maps, src, pairs, tile=tile, grid=g) for g in (0, 456)], w.poses


@pytest.mark.parametrize("sizes,tile", [
    ([1, 31, 33, 255], 16384), ([256, 257, 2047, 2049], 16384), ([4095, 4097, 16383, 16385], 16384),
    ([20000, 33000, 5000, 12345], 16384), ([9000, 7001, 2048, 3], 2048), ([30011, 29000, 1, 40], 4096),
    ([114 * 2048 - 4, 1, 1, 1], 2048),
])
def test_same_sums_as_the_per_point_kernel(dev, sizes, tile):  # noqa: F811
    (a, b), poses = _plans(sizes, tile)
    P = len(poses)
    base = torch.tensor(poses, device="cuda")
    xi = torch.tensor(1e-3 * np.random.default_rng(1).normal(size=(P, 6)), device="cuda")
    ra, rb = a.execute(poses), b.execute(poses)
    assert torch.equal(ra.out, rb.out) and torch.equal(ra.inliers, rb.inliers)
    assert int(ra.inliers.sum()) > 0
    for mode in (1, 2, 3):
        ga, na = a.evaluate(base, xi, mode=mode)
        gb, nb = b.evaluate(base, xi, mode=mode)
        assert torch.equal(ga, gb) and torch.equal(na, nb)


def test_points_without_a_voxel_and_not_finite(dev):  # noqa: F811
    (a, b), poses = _plans([5000, 5000, 5000, 5000], 16384, seed=4)
    for p in (a, b):
        for pts, _ in p._refs[1]:
            pts[::7] += 1e4                    # no voxel there
            pts[5] = float("inf")
            pts[6] = float("nan")
    ra, rb = a.execute(poses), b.execute(poses)
    assert bool(torch.isfinite(ra.out).all())
    assert torch.equal(ra.out, rb.out) and torch.equal(ra.inliers, rb.inliers)


@pytest.mark.parametrize("n,tile", [(0, 0), (1, 0), (31, 0), (255, 0), (256, 0), (257, 0), (2048, 0),
                                    (8191, 0), (8192, 0), (8193, 0), (16384, 0), (16385, 0),
                                    (16385, 512), (32768, 512), (32769, 512), (700, 100)])
def test_single_factor_in_one_launch(dev, n, tile):  # noqa: F811
    """A small single factor is one cluster's work; a grid request keeps the general
    launches.  Same sums, with the scratch of vgicp_linearize and without allocation."""
    w = synth.with_surface_covariances(
        synth.outdoor_submaps(seed=8, n_submaps=2, n_min=33000, n_max=33000, neighbours=1))
    (tp, tc), (sp, sc) = w.clouds.cloud(int(w.pairs[0, 0])), w.clouds.cloud(int(w.pairs[0, 1]))
    vm = api.VoxelMap.build(cu(tp), cu(tc), 1.0)
    src = (cu(sp[:n]), cu(sc[:n]))
    a = api.linearize(vm, *src, w.poses[0], tile=tile)
    b = api.linearize(vm, *src, w.poses[0], tile=tile, grid=456)
    assert torch.equal(a.out, b.out) and torch.equal(a.inliers, b.inliers)
    if n > 100:
        assert int(a.inliers) > 0
