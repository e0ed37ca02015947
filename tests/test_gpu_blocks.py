"""27 neighbours from occupancy blocks (batched calls of a million source points and
more) against the kernel that probes voxel by voxel (plans): the same terms in the
same order, so results must be equal bit for bit.  Scenes: surfaces, a filled volume
(full blocks), isolated voxels (one per block: more blocks than a quarter of the
voxels), maps rebuilt with many more voxels than their first build (no room: left to the
probes) beside maps that fit, and keys at both ends of the range."""
import numpy as np
import pytest
import torch

from paper_2202_00242_gb300 import api, synth

from test_gpu_parity import cu, dev  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

N = 60000
R = 0.5


def _scene(kind, seed):
    rng = np.random.default_rng(seed)
    if kind == "surface":
        w = synth.with_surface_covariances(
            synth.outdoor_submaps(seed=seed, n_submaps=2, n_min=N, n_max=N, neighbours=1))
        return w.clouds.cloud(0)
    if kind == "volume":
        p = rng.uniform(-8.0, 8.0, (N, 3))
    elif kind == "isolated":
        k = rng.choice(120 ** 3, N // 8, replace=False)
        c = np.stack([k % 120, k // 120 % 120, k // 14400], 1) * 4.0 - 240.0
        p = (c[rng.integers(0, len(c), N)] + rng.uniform(0.1, 0.9, (N, 3))) * R
    else:  # "ends": voxels at both ends of the key range and around zero
        k = rng.choice([-(1 << 20), -(1 << 20) + 1, -2, -1, 0, 1, (1 << 20) - 2, (1 << 20) - 1],
                       (N, 3)).astype(np.float64)
        p = (k + rng.uniform(0.25, 0.75, (N, 3))) * R
    c = np.tile(np.array([0.02, 0.001, 0, 0.03, 0, 0.02], np.float32), (N, 1))
    return p.astype(np.float32), c


def _compare(maps, sources, seed, modes=True):
    rng = np.random.default_rng(seed)
    pairs = np.array([[j % len(maps), i % len(sources)] for i in range(20) for j in (0, i)], np.int32)
    poses = np.stack([synth.perturb_pose(rng, np.eye(4), 0.2, 0.0 if i % 3 else 2.0)
                      for i in range(len(pairs))])
    got = api.linearize_batched(maps, sources, pairs, poses, neighbours=27)
    plan = api.Plan(maps, sources, pairs, neighbours=27)
    want = plan.execute(poses)
    assert int(want.inliers.sum()) > 0
    assert torch.equal(got.inliers, want.inliers) and torch.equal(got.out, want.out)
    if modes:
        base = torch.tensor(poses, device="cuda")
        for mode in (1, 2, 3):
            g, e, n = api.evaluate_batched(maps, sources, pairs, poses, mode=mode, neighbours=27)
            o, m = plan.evaluate(base, mode=mode)
            assert torch.equal(n, m) and torch.equal(e, o[:, 6])
            if mode > 1:
                assert torch.equal(g, o[:, :6])


@pytest.mark.parametrize("kind", ["surface", "volume", "isolated", "ends"])
def test_same_as_the_probes(dev, kind):  # noqa: F811
    clouds = [_scene(kind, s) for s in (1, 2)]
    maps = [api.VoxelMap.build(cu(p), cu(c), R) for p, c in clouds]
    for m in maps:
        m.status()
    _compare(maps, maps, 3)
    _compare(maps, [(cu(p), cu(c)) for p, c in clouds], 4, modes=False)


def test_maps_that_outgrew_their_first_build(dev):  # noqa: F811
    small = np.tile(np.array([[0.1, 0.1, 0.1], [0.7, 0.1, 0.1]], np.float32), (N // 2, 1))
    cov = np.tile(np.array([0.02, 0, 0, 0.03, 0, 0.02], np.float32), (N, 1))
    full = [_scene("surface", s) for s in (5, 6)]
    maps = [api.VoxelMap.build(cu(small), cu(cov), R), api.VoxelMap.build(cu(full[0][0]), cu(full[0][1]), R)]
    api.rebuild_voxelmaps([maps[0]], cu(full[1][0]), cu(full[1][1]))  # 2 voxels -> thousands
    for m in maps:
        m.status()
    _compare(maps, maps, 7)
