"""Voxel keys of transformed source points where the float32 fast path changes
course: on and next to faces, at both ends of the key range, beyond the range of the
fast path (2^22 voxels), at infinity and NaN.  Keys must equal the binary64
definition, correspondences and counts the target's voxels, with 1 and with 27
neighbours, and the results must not depend on whether the debug outputs are written."""
import numpy as np
import pytest
import torch

from paper_2202_00242_gb300 import api

from test_gpu_parity import cu, dev  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

R = 0.25
TOP = float(1 << 20)


def _sources():
    rng = np.random.default_rng(3)
    edge = []
    for k in (-TOP - 2, -TOP - 1, -TOP, -TOP + 1, -3, -1, 0, 1, 2, TOP - 2, TOP - 1, TOP, TOP + 1,
              2 * TOP, 4 * TOP - 1, 4 * TOP, -4 * TOP, 2.0 ** 31, -2.0 ** 33, 1e30):
        for eps in (0.0, 0.5, 1e-4, -1e-4):
            edge.append([(k + eps) * R, 0.1, -0.1])
            edge.append([0.1, (k + eps) * R, 0.1])
            edge.append([-0.1, 0.1, (k + eps) * R])
    edge += [[-0.0, -0.0, 0.0], [np.inf, 0, 0], [0, -np.inf, 0], [0, 0, np.nan], [np.nan] * 3]
    near = rng.uniform(-1.0, 1.0, (600, 3))
    near[:200] = np.round(near[:200] / R) * R + rng.choice([0, 1e-7, -1e-7, 3e-6], (200, 3))
    return np.concatenate([np.array(edge), near]).astype(np.float32)


@pytest.mark.parametrize("neighbours", [1, 27])
@pytest.mark.parametrize("shift", [0.0, 0.125])
def test_keys_and_counts(dev, neighbours, shift):  # noqa: F811
    src = _sources()
    rng = np.random.default_rng(4)
    tgt = np.concatenate([rng.uniform(-1.2, 1.2, (400, 3)),
                          [[(-TOP + .5) * R, .1, -.1], [(TOP - .5) * R, .1, -.1],
                           [.1, (TOP - .5) * R, .1], [-.1, .1, (-TOP + .5) * R]]]).astype(np.float32)
    iso = np.array([0.02, 0, 0, 0.02, 0, 0.02], np.float32)
    vm = api.VoxelMap.build(cu(tgt), cu(np.tile(iso, (len(tgt), 1))), R)
    vm.status()
    occupied = {tuple(k) for k in vm.export()["keys"]}
    T = np.eye(4)
    T[:3, 3] = shift
    P, C = cu(src), cu(np.tile(iso, (len(src), 1)))
    dbg = api.linearize(vm, P, C, T, neighbours=neighbours, corr=True, qkeys=True)
    rel = api.linearize(vm, P, C, T, neighbours=neighbours)
    with np.errstate(invalid="ignore"):
        keys = np.floor((src.astype(np.float64) + shift) / R)
    ok = np.all(np.abs(keys) < 2.0 ** 30, axis=1)  # finite, and far from the int range's ends
    assert np.array_equal(dbg.qkeys.cpu().numpy()[ok], keys[ok].astype(np.int64))
    offsets = [(0, 0, 0)] if neighbours == 1 else [
        (x, y, z) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)]
    want, own = 0, []
    for k in keys:
        fine = bool(np.all(np.abs(k) < 2.0 ** 40))
        near = [tuple(int(v) + d for v, d in zip(k, o)) for o in offsets] if fine else []
        want += sum(n in occupied for n in near)
        own.append(fine and tuple(int(v) for v in k) in occupied)
    assert int(rel.inliers) == int(dbg.inliers) == want and want > 0
    assert np.array_equal(dbg.corr.cpu().numpy() >= 0, np.array(own))
    assert torch.equal(rel.out, dbg.out)
