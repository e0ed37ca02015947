"""Neighbour lists where squared distances differ by a few float32 steps: shells of
neighbours at nearly one distance (six around a point, and the shells of a jittered cubic
lattice), at list lengths well below the number of candidates the search keeps.  Such
values share the leading bits by which they are first selected, so the order within a
shell, and which of it are the k nearest, has to come from the full values.  Lists must
equal the oracle's exactly (binary64 squared distance, then index)."""
import numpy as np
import pytest

import oracle
from paper_2202_00242_gb300 import api

from test_gpu_parity import cu, dev  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _check(pts, off, k, cell):
    _, nbr = api.estimate_covariances(cu(pts), offsets=off, k=k, cell=cell, neighbours=True)
    nbr = nbr.cpu().numpy().astype(np.int64)
    for a, b in zip(off[:-1], off[1:]):
        assert np.array_equal(nbr[a:b], oracle.knn_bruteforce(pts[a:b], k)), (a, k)


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 6, 7])
def test_six_neighbours_at_nearly_one_distance(dev, k):  # noqa: F811
    rng = np.random.default_rng(k)
    clouds = []
    for _ in range(300):
        d = 0.9 * (1.0 + rng.uniform(-1.0, 1.0, 6) * 2.0 ** -16)
        axes = np.concatenate([np.eye(3), -np.eye(3)]) * d[:, None]
        p = 0.5 + np.concatenate([np.zeros((1, 3)), axes])
        clouds.append(p[np.concatenate([[0], 1 + rng.permutation(6)])])
    pts = np.concatenate(clouds).astype(np.float32)
    _check(pts, np.arange(301) * 7, k, 1.0)


@pytest.mark.parametrize("k", [2, 3, 4, 5, 6, 7, 8, 11, 12, 13, 14, 15, 16, 17, 18, 24, 28])
@pytest.mark.parametrize("jitter", [2.0 ** -18, 2.0 ** -15])
def test_jittered_lattice(dev, k, jitter):  # noqa: F811
    rng = np.random.default_rng(k)
    g = np.stack(np.meshgrid(*[np.arange(9)] * 3, indexing="ij"), -1).reshape(-1, 3)
    pts = (0.25 * g[rng.permutation(len(g))] + rng.uniform(-jitter, jitter, (len(g), 3))).astype(np.float32)
    _check(pts, np.array([0, len(pts)]), k, 0.0)
    _check(pts, np.array([0, len(pts)]), k, 0.3)
