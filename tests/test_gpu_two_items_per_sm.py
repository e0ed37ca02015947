"""Sets of up to two work items per SM, too many for a cluster each, go to a kernel with
two or four points per thread in flight; any grid request keeps the per-point kernel.  Each
thread adds the same float32 terms in the same order, so H, b, err, the gradients and
the counts must be equal bit for bit, at ragged sizes (items of one point, whole rounds,
a round and a point, tails of warps) and on both sides of the limits."""
import numpy as np
import pytest
import torch

from paper_2202_00242_gb300 import api, synth

from test_gpu_parity import cu, dev  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _plans(sizes, tile):
    w = synth.with_surface_covariances(
        synth.outdoor_submaps(seed=11, n_submaps=len(sizes), n_min=max(sizes), n_max=max(sizes),
                              neighbours=1))
    clouds = [w.clouds.cloud(c) for c in range(len(sizes))]
    maps = [api.VoxelMap.build(cu(p), cu(c), 1.0) for p, c in clouds]
    src = [(cu(p[:n]), cu(c[:n])) for (p, c), n in zip(clouds, sizes)]
    return [api.Plan(maps, src, w.pairs, tile=tile, grid=g) for g in (0, 456)], w.poses


def _same(a, b, poses):
    base = torch.tensor(poses, device="cuda")
    xi = torch.tensor(1e-3 * np.random.default_rng(1).normal(size=(len(poses), 6)), device="cuda")
    ra, rb = a.execute(poses), b.execute(poses)
    assert torch.equal(ra.out, rb.out) and torch.equal(ra.inliers, rb.inliers)
    assert int(ra.inliers.sum()) > 0
    for mode in (1, 2, 3):
        ga, na = a.evaluate(base, xi, mode=mode)
        gb, nb = b.evaluate(base, xi, mode=mode)
        assert torch.equal(ga, gb) and torch.equal(na, nb)


# items of 152 SMs: 58 is the first set too large for clusters, 152 and 304 the last
# with one and two items per SM
@pytest.mark.parametrize("sizes,tile", [
    ([55 * 2048 + 1, 1, 31], 2048),                       # 58 items, three of one warp
    ([80 * 2048 + 1024, 70 * 2048 + 1025, 511], 2048),    # 153 items: one round and a point more
    ([80 * 2048 + 512, 69 * 2048 + 513, 767], 2048),      # 152 items: two rounds, tails of them
    ([61 * 2560 + 255, 50 * 2560 + 257, 2559], 2560),     # ten points per thread
    ([152 * 2048, 100 * 2048 + 33, 51 * 2048], 2048),     # 304 items
    ([152 * 2048, 100 * 2048 + 33, 51 * 2048 + 1], 2048),  # 305 items
])
def test_same_sums_as_the_per_point_kernel(dev, sizes, tile):  # noqa: F811
    (a, b), poses = _plans(sizes, tile)
    _same(a, b, poses)


def test_points_without_a_voxel_and_not_finite(dev):  # noqa: F811
    (a, b), poses = _plans([180001, 120003, 30007], 2048)
    for pts, _ in a._refs[1]:
        pts[::7] += 1e4                    # no voxel there
        pts[5] = float("inf")
        pts[6] = float("nan")
    _same(a, b, poses)
    assert bool(torch.isfinite(a.execute(poses).out).all())


@pytest.mark.parametrize("sizes", [[5000, 3000, 1], [130 * 2048, 9, 9]])
def test_execution_without_a_status_word(dev, sizes):  # noqa: F811
    """Where every item has a CTA an execution clears and reads no status word: what an
    evaluation at a pose that is not finite left there does not reach it."""
    (a, b), poses = _plans(sizes, 2048)
    base = torch.tensor(poses, device="cuda")
    xi = torch.zeros((len(poses), 6), dtype=torch.float64, device="cuda")
    want = b.execute(poses)
    for p in (a, b):
        p.execute(poses)                   # captures
        xi[0, 0] = float("nan")
        g, n = p.evaluate(base, xi, mode=2)
        assert bool(torch.isnan(g).all()) and bool((n == -1).all())
        got = p.execute(poses)
        assert torch.equal(got.out, want.out) and torch.equal(got.inliers, want.inliers)
