"""The k-NN search kernels at the sizes where they change course: cells of one
query to a warp's worth, neighbourhoods of more candidates than one tile (192) and
than the first kernel takes (512), ties beyond the collecting list (64), clouds
around the queries-per-warp limits, every list length, outliers far from any
cell, and coordinates near the edge of the key range.  Neighbour lists must equal
the oracle's exactly (binary64 squared distance, then index); covariances are
compared as in test_gpu_knn (2e-5 where the smallest eigenvalue is separated)."""
import numpy as np
import pytest

from test_gpu_knn import _check
from test_gpu_parity import dev  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _surface(n, seed, size=20.0):
    rng = np.random.default_rng(seed)
    p = rng.uniform(0.0, size, (n, 3))
    p[:, 2] = 0.02 * rng.normal(size=n) + np.where(rng.random(n) < 0.3, 3.0, 0.0)
    return p.astype(np.float32)


@pytest.mark.parametrize("k", [1, 2, 9, 10, 11, 19, 20, 21, 31, 32])
def test_list_lengths(dev, k):  # noqa: F811
    _check(_surface(3000, k), k=k)


@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 31, 33, 129, 24319, 24321])
def test_cloud_sizes(dev, n):  # noqa: F811
    _check(_surface(n, n), k=10)


@pytest.mark.parametrize("cell", [0.05, 1.1, 3.0, 30.0])
def test_candidates_per_block(dev, cell):  # noqa: F811
    # 2,500 points on 20 x 20 m: from less than one to all points per cell
    _check(_surface(2500, 5), k=10, cell=cell)


def test_ties_beyond_the_list(dev):  # noqa: F811
    p = _surface(1500, 6)
    p[100:300] = p[100]                       # 200 copies of one point
    p[300:340] = p[300]                       # 40 of another
    rng = np.random.default_rng(1)
    ring = np.repeat(np.array([[1, 0, 0], [-1, 0, 0], [0, 1, 0], [0, -1, 0]]), 25, axis=0)
    p = np.concatenate([p, (50.0 + ring).astype(np.float32)])[rng.permutation(1600)]
    _check(p, k=10)
    _check(p, k=32)


def test_outliers_and_large_coordinates(dev):  # noqa: F811
    p = _surface(4000, 7)
    p[5] = (400.0, -300.0, 250.0)             # far outside
    p[6] = (-900.0, 10.0, 0.0)
    _check(p, k=10, cell=0.5)
    _check(p, k=10)
    _check(p + np.float32(30000.0), k=10)
