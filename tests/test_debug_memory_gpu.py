"""sgmf_debug_stage with little host memory left: the volumes leave the device
through a buffer of bounded size, and no C++ exception crosses the C boundary.
In a process of its own, whose address space is limited to 48 MiB above what it
holds (the volumes are 75 and 150 MiB)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

_CHILD = r"""
import resource, sys
sys.path.insert(0, sys.argv[1])
import numpy as np, torch
from paper_2504_05148_gb300 import scenes, sgmf as S
s = scenes.random_small(31, 640, 480, 256)
ctx = S.Context(s.W, s.H, s.D)
ctx.set_debug(True)
out = torch.empty(s.shape, dtype=torch.int16, device="cuda")
ctx.compute(*(torch.from_numpy(a).cuda() for a in (s.left, s.right, s.lidar)), out)
stages = (S.SGMF_STAGE_COST, S.SGMF_STAGE_SUM, S.SGMF_STAGE_CENSUS_L)
want = [ctx.stage(i) for i in stages]
got = [np.zeros_like(a) for a in want]
for g in got:
    g.fill(1)
held = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
resource.setrlimit(resource.RLIMIT_AS, (held + (48 << 20), resource.RLIM_INFINITY))
for i, g in zip(stages, got):
    S.sgmf_debug_stage(ctx.handle, i, g.ctypes.data, g.nbytes)
resource.setrlimit(resource.RLIMIT_AS, (resource.RLIM_INFINITY, resource.RLIM_INFINITY))
assert all((g == w).all() for g, w in zip(got, want))
ctx.close()
print("same")
"""


def test_volumes_leave_through_a_bounded_buffer(gpu):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _CHILD, root], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "same" in r.stdout, (r.returncode, r.stderr[-2000:])
