"""Downsampling at the sizes where it changes course: one point, whole words of the
first-point bitmap, groups of up to and over 8 points and of thousands, sums that
round in double-float (very different magnitudes in one voxel), empty clouds, and more
points than one CTA scans.  Everything must equal the oracle bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2202_00242_gb300 import api

from test_gpu_parity import cu, dev  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _check(pts, t, r, split, sizes=None):
    off = np.concatenate([[0], np.cumsum(sizes if sizes is not None else [len(pts)])])
    gp, gt, gc, oo = api.downsample(cu(pts), r, times=None if t is None else cu(t), split=split,
                                    offsets=off)
    gp, gc = gp.cpu().numpy(), gc.cpu().numpy()
    for c in range(len(off) - 1):
        a, b = off[c], off[c + 1]
        rp, rt, rc = oracle.downsample(pts[a:b], None if t is None else t[a:b], r, split)
        o = slice(oo[c], oo[c + 1])
        assert oo[c + 1] - oo[c] == len(rc)
        assert np.array_equal(gc[o], rc) and np.array_equal(gp[o], rp)
        if t is not None:
            assert np.array_equal(gt.cpu().numpy()[o], rt)


def _cloud(n, extent, seed):
    rng = np.random.default_rng(seed)
    return (rng.uniform(-extent, extent, (n, 3)).astype(np.float32),
            np.sort(rng.random(n)).astype(np.float32))


@pytest.mark.parametrize("n,extent", [(1, 1.0), (31, 2.0), (32, 2.0), (33, 2.0), (256, 3.0),
                                      (257, 3.0), (4096, 1.0), (9000, 0.6), (20011, 12.0)])
@pytest.mark.parametrize("split", [0.0, 0.2])
def test_sizes(dev, n, extent, split):  # noqa: F811
    pts, t = _cloud(n, extent, n)
    _check(pts, t, 0.5, split)
    _check(pts, None, 0.5, 0.0)


def test_inexact_sums(dev):  # noqa: F811
    pts, t = _cloud(6000, 0.9, 1)
    pts *= np.float32(10.0) ** np.random.default_rng(2).integers(-9, 1, pts.shape).astype(np.float32)
    _check(pts, t, 1.0, 0.3)


def test_many_clouds(dev):  # noqa: F811
    sizes = [0, 700, 0, 1, 2500, 33, 0]
    pts, t = _cloud(sum(sizes), 4.0, 3)
    _check(pts, t, 0.7, 0.1, sizes)


def test_more_points_than_one_cta_scans(dev):  # noqa: F811
    pts, t = _cloud(16384 * 32 + 77, 30.0, 4)
    _check(pts, t, 0.8, 0.25)
