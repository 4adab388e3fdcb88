"""fvna_step_noalloc takes device memory in its first call on a device at most:
later calls, whatever their limiter, size or geometry, leave the free memory
as it is.  In a process of its own, where no other entry point has loaded a
kernel before."""
import subprocess
import sys

import pytest

from conftest import ROOT

pytestmark = pytest.mark.gpu

CHILD = """
import torch
from paper_1311_3004_gb300 import build, fvna
build.build()
torch.zeros(1, device="cuda")
calls = []
for lim in (fvna.LIM_MC, fvna.LIM_NONE, fvna.LIM_LW):
    for geometry in (fvna.CARTESIAN, fvna.AXISYMMETRIC):
        for nx, ny in ((64, 64), (700, 700), (20000, 8)):
            q = torch.zeros((3, ny, nx), dtype=torch.float64, device="cuda")
            q[0] = 1.0
            q[0, ny // 2, nx // 2] += 1e-3
            cfg = fvna.make_config(precision=fvna.FP64, limiter=lim, geometry=geometry, beta=3.5,
                                   delta=1e-3, dx=1.0 / 32, dt_fixed=0.01)
            calls.append((cfg, fvna.make_domain(nx, ny), q, torch.empty_like(q)))
torch.cuda.synchronize()
free = None
for cfg, dom, a, b in calls:
    assert fvna.step_noalloc(cfg, dom, a, b, 0.0, 0.01)[0] == fvna.OK
    now = torch.cuda.mem_get_info()[0]
    if free is None:
        free = now
    assert now == free, (cfg.limiter, dom.nx, dom.ny, free - now)
print("same")
"""


def test_only_the_first_call_sets_up():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0 and r.stdout.strip().endswith("same"), r.stderr[-2000:]
