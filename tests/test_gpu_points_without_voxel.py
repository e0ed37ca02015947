"""Batches with points that have no voxel (NaN, or outside the key range): a few, half and
all of a map's, in the first, a middle and the last map, in maps of a few points each, and
in sets of both finalize kernels.  The build reports them, and leaves them out: every
voxel's key, count, mean and covariance is that of the map's other points bit for bit,
the grouped cloud holds those points and NaN rows behind them, and the factors see just
the points that are left.  First builds, rebuilds, and sound rebuilds after them."""
import numpy as np
import pytest
import torch

import oracle
from paper_2202_00242_gb300 import api
from paper_2202_00242_gb300._lib import VGICPError

from test_gpu_parity import cu, dev  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

R = 0.5


def _clouds(sizes, extent, seed):
    rng = np.random.default_rng(seed)
    n = int(sum(sizes))
    pts = rng.uniform(-extent, extent, (n, 3)).astype(np.float32)
    return pts, rng.uniform(0.5, 1.0, (n, 6)).astype(np.float32)


def _spoil(pts, a, b, part, seed):
    rng = np.random.default_rng(seed)
    bad = a + rng.permutation(b - a)[:max(1, int(round(part * (b - a))))]
    pts[bad, rng.integers(0, 3, len(bad))] = rng.choice([np.nan, np.inf, 3.0e7], len(bad))
    return bad


def _check(maps, pts, covs, off, report):
    if report:
        with pytest.raises(VGICPError) as e:
            maps[0].status()
        assert e.value.code == -4
    else:
        maps[0].status()
    good = np.all(np.abs(pts) < 1.0e5, axis=1)
    for m, vm in enumerate(maps):
        p, c, ok = (x[off[m]:off[m + 1]] for x in (pts, covs, good))
        p, c = p[ok], c[ok]
        ref, ex = oracle.build_voxelmap(p, c, R), vm.export()
        assert np.array_equal(ex["keys"], ref.keys), m
        assert np.array_equal(ex["counts"], ref.counts), m
        assert np.array_equal(ex["means"], ref.means.astype(np.float32)), m
        assert np.array_equal(ex["covs"], ref.covs.astype(np.float32)), m
        g, gc = (x.cpu().numpy() for x in vm.grouped_cloud())
        k = len(p)
        assert np.isnan(g[k:]).all() and np.isnan(gc[k:]).all(), m
        rows, inp = np.concatenate([g[:k], gc[:k]], 1), np.concatenate([p, c], 1)
        where = {r.tobytes(): i for i, r in enumerate(inp)}
        idx = np.array([where[r.tobytes()] for r in rows], np.int64)
        assert np.array_equal(np.sort(idx), np.arange(k)), m
        key = np.floor(g[:k].astype(np.float64) / R)
        same = np.all(key[1:] == key[:-1], axis=1)
        assert np.all(idx[1:][same] > idx[:-1][same]), m
        assert int((~same).sum()) + (k > 0) == len(ref.counts), m


def _run(sizes, extent, spoiled, seed):
    """spoiled: (map, part of its points) pairs."""
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    pts, covs = _clouds(sizes, extent, seed)
    other, oc = _clouds(sizes, extent, seed + 1)
    bad = pts.copy()
    for j, (m, part) in enumerate(spoiled):
        _spoil(bad, off[m], off[m + 1], part, seed + j)
    first = api.build_voxelmaps(cu(bad), cu(covs), off, R)
    _check(first, bad, covs, off, True)
    maps = api.build_voxelmaps(cu(other), cu(oc), off, R)
    for p, c, report in ((bad, covs, True), (bad, covs, True), (pts, covs, False),
                         (other, oc, False), (bad, covs, True)):
        api.rebuild_voxelmaps(maps, cu(p), cu(c))
        _check(maps, p, c, off, report)
    # a map as source: its cloud without the points that have no voxel
    good = np.all(np.abs(bad) < 1.0e5, axis=1)
    pairs = [[(m + 1) % len(sizes), m] for m in range(len(sizes))]
    T = np.tile(np.eye(4), (len(pairs), 1, 1))
    got = api.linearize_batched(maps, maps, pairs, T)
    assert bool(torch.isfinite(got.out).all())
    occupied = [{tuple(k) for k in vm.export()["keys"]} for vm in maps]
    for i, (t, s) in enumerate(pairs):
        q = bad[off[s]:off[s + 1]][good[off[s]:off[s + 1]]].astype(np.float64)
        want = sum(tuple(k) in occupied[t] for k in np.floor(q / R).astype(np.int64))
        assert int(got.inliers[i]) == want


@pytest.mark.parametrize("part", [0.001, 0.5, 1.0])
@pytest.mark.parametrize("which", [0, 1, 3])
def test_one_map_of_four(dev, part, which):  # noqa: F811
    _run([3000, 4001, 700, 2500], 6.0, [(which, part)], 11)


@pytest.mark.parametrize("part", [0.1, 0.7, 1.0])
def test_every_map(dev, part):  # noqa: F811
    _run([900, 1500, 1, 640], 4.0, [(m, part) for m in range(4)], 12)


@pytest.mark.parametrize("extent", [1.0, 30.0])
def test_neighbouring_maps_without_a_voxel(dev, extent):  # noqa: F811
    _run([800, 50, 0, 60, 900, 0, 70], extent, [(1, 1.0), (3, 1.0), (4, 0.3), (6, 1.0)], 13)


@pytest.mark.parametrize("extent", [0.6, 3.0])
def test_maps_of_a_few_points(dev, extent):  # noqa: F811
    sizes = np.random.default_rng(5).integers(0, 40, 60)
    sizes[7], sizes[30] = 5, 33
    spoiled = [(m, (0.2, 0.5, 1.0)[m % 3]) for m in range(0, 60, 4) if sizes[m]] + [(7, 1.0), (30, 0.9)]
    _run(list(sizes), extent, spoiled, 14)


@pytest.mark.parametrize("extent,part", [(0.7, 0.3), (4.0, 0.02)])
def test_long_lists_before_a_gap(dev, extent, part):  # noqa: F811
    _run([9000, 6000, 5000], extent, [(0, part), (1, part)], 15)


def test_large_set_of_short_lists(dev):  # noqa: F811
    sizes = [130000, 5, 200000, 90000, 100000]
    _run(sizes, 18.0, [(0, 0.4), (1, 1.0), (3, 0.0001), (4, 1.0)], 16)
