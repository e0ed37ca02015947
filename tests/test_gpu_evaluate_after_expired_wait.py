"""A plan whose graph ran out of a wait of the staged kernel, and its evaluations after
that: they start from clean state, so the first one, the second one, and an execution
between them are those of a plan that never failed.

The wait hook arms one launch, and a plan's first execution launches twice (once before
it records its graph), so a host thread keeps the hook armed until the graph holds an
expiring launch; its waits end after 20 ms."""
import threading
import time

import numpy as np
import pytest
import torch

from paper_2202_00242_gb300 import _lib, api, synth

from test_gpu_parity import cu, dev  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [1, 2, 3])
def test_evaluation_after_an_expired_execution(dev, mode):  # noqa: F811
    lib = _lib.load()
    w = synth.with_surface_covariances(
        synth.outdoor_submaps(seed=17, n_submaps=3, n_min=5000, n_max=5000, neighbours=1))
    clouds = [w.clouds.cloud(c) for c in range(3)]
    maps = [api.VoxelMap.build(cu(p), cu(c), 1.0) for p, c in clouds]
    srcs = [(cu(p), cu(c)) for p, c in clouds]
    base = torch.tensor(w.poses, device="cuda")
    xi = torch.tensor(1e-3 * np.random.default_rng(2).normal(size=(len(w.pairs), 6)), device="cuda")
    want, want_n = api.Plan(maps, srcs, w.pairs, variant=2).evaluate(base, xi, mode=mode)
    assert bool(torch.isfinite(want[:, 6]).all())
    plan = api.Plan(maps, srcs, w.pairs, variant=2)
    stop = threading.Event()

    def keep_armed():
        while not stop.is_set():
            lib.vgicp_test_expire_waits(0, 20_000_000)
            time.sleep(1e-3)

    lib.vgicp_test_expire_waits(0, 20_000_000)
    t = threading.Thread(target=keep_armed)
    t.start()
    try:
        bad = plan.execute(w.poses)
        torch.cuda.synchronize()
    finally:
        stop.set()
        t.join()
    # use up the hook, which may still be armed
    api.linearize(maps[0], *srcs[0], np.eye(4), variant=2, tile=1024)
    torch.cuda.synchronize()
    assert bool(torch.isnan(bad.out).all()) and bool((bad.inliers == -1).all())
    for _ in range(2):
        got, got_n = plan.evaluate(base, xi, mode=mode)
        assert torch.equal(got, want) and torch.equal(got_n, want_n)
    plan.execute(w.poses)  # expires again
    got, got_n = plan.evaluate(base, xi, mode=mode)
    assert torch.equal(got, want) and torch.equal(got_n, want_n)
    xi[0, 1] = float("nan")
    got, got_n = plan.evaluate(base, xi, mode=mode)
    assert bool(torch.isnan(got).all()) and bool((got_n == -1).all())
