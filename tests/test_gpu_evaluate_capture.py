"""A differentiable evaluation recorded in a caller's CUDA graph: a replay at a pose that is
not finite gives NaN, and the next replay at finite poses is sound again."""
import numpy as np
import pytest
import torch

from paper_2202_00242_gb300 import api, synth

from test_gpu_parity import cu, dev  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [1, 2, 3])
def test_replay_after_a_pose_that_is_not_finite(dev, mode):  # noqa: F811
    w = synth.with_surface_covariances(
        synth.outdoor_submaps(seed=13, n_submaps=3, n_min=5000, n_max=5000, neighbours=1))
    clouds = [w.clouds.cloud(c) for c in range(3)]
    maps = [api.VoxelMap.build(cu(p), cu(c), 1.0) for p, c in clouds]
    plan = api.Plan(maps, [(cu(p), cu(c)) for p, c in clouds], w.pairs)
    base = torch.tensor(w.poses, device="cuda")
    good = torch.tensor(1e-3 * np.random.default_rng(2).normal(size=(3, 6)), device="cuda")
    xi = good.clone()
    want, want_n = (t.clone() for t in plan.evaluate(base, good, mode=mode))
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        g, n = plan.evaluate(base, xi, mode=mode)
    for _ in range(2):
        graph.replay()
        assert torch.equal(g, want) and torch.equal(n, want_n)
        xi[1, 2] = float("inf")
        graph.replay()
        assert bool(torch.isnan(g).all()) and bool((n == -1).all())
        xi.copy_(good)
