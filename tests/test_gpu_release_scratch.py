"""The scratch that the library keeps between calls goes back to the device: by
release_scratch in a program that has no map (k-NN covariances and downsampling only),
by itself with the last map.  In a process of its own, where nothing else holds memory."""
import os
import subprocess
import sys

import pytest

from test_gpu_parity import dev  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

PROGRAM = """
import torch
from paper_2202_00242_gb300 import api

def free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0] >> 20

def calls(p):
    api.estimate_covariances(p, k=10)
    api.downsample(p, 0.5)

p = torch.rand((1500000, 3), device="cuda") * 100.0
calls(p[:1000].contiguous())          # modules loaded
api.release_scratch()
start = free()
calls(p)
kept = start - free()
api.release_scratch()
left = start - free()
calls(p)                              # and the scratch can be taken anew
c = torch.tensor([1.0, 0, 0, 1, 0, 1], device="cuda").repeat(1000, 1)
vm = api.VoxelMap.build(p[:1000].contiguous(), c, 1.0)
vm.status()
vm.close()
by_map = start - free()
print("MB", kept, left, by_map)
"""


def test_scratch_goes_back(dev):  # noqa: F811
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=root, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stderr
    kept, left, by_map = (int(x) for x in r.stdout.split("MB")[1].split())
    # 1.5M points take more than 100 bytes each of scratch; the rest is rounding
    assert kept > 100 and left < 16 and by_map < 16, r.stdout
