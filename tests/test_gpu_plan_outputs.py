"""Where a plan's execution puts its results: buffers that a kernel cannot store doubles to
(device memory at an odd multiple of four bytes) get them by a copy, byte for byte what
aligned ones hold; either buffer may be null."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2202_00242_gb300 import _lib, api, synth

from test_gpu_parity import cu, dev  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("out_shift,inl_shift", [(0, 0), (4, 0), (0, 4), (4, 4), (1, 2)])
def test_unaligned_buffers(dev, out_shift, inl_shift):  # noqa: F811
    w = synth.with_surface_covariances(
        synth.outdoor_submaps(seed=23, n_submaps=3, n_min=5000, n_max=5000, neighbours=1))
    clouds = [w.clouds.cloud(c) for c in range(3)]
    maps = [api.VoxelMap.build(cu(p), cu(c), 1.0) for p, c in clouds]
    plan = api.Plan(maps, [(cu(p), cu(c)) for p, c in clouds], w.pairs)
    want = plan.execute(w.poses)
    n = len(w.pairs)
    poses = np.ascontiguousarray(w.poses, dtype=np.float64)

    def run(out, inl):
        _lib.check(_lib.load().vgicp_plan_execute(
            plan._h, poses.ctypes.data_as(ctypes.c_void_p), out, inl, None, None,
            api._stream_ptr()))
        torch.cuda.synchronize()

    ob = torch.zeros(8 * 43 * n + 16, dtype=torch.uint8, device="cuda")
    ib = torch.zeros(8 * n + 16, dtype=torch.uint8, device="cuda")
    op, ip = ctypes.c_void_p(ob.data_ptr() + out_shift), ctypes.c_void_p(ib.data_ptr() + inl_shift)
    for o, i in ((op, ip), (op, None), (None, ip)):
        ob.zero_()
        ib.zero_()
        run(o, i)
        got = ob.cpu().numpy()[out_shift:out_shift + 8 * 43 * n].tobytes()
        assert got == (want.out.cpu().numpy().tobytes() if o else bytes(len(got)))
        got = ib.cpu().numpy()[inl_shift:inl_shift + 8 * n].tobytes()
        assert got == (want.inliers.cpu().numpy().tobytes() if i else bytes(len(got)))
