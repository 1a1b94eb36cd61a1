"""The first forward of a process loads device code: its cost beside a repeated one."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHILD = """
import time, torch
from paper_2607_19378_b200 import hyenand as hn
q, k, v = torch.randn(3, 1, 8, 512, 512, device="cuda").unbind(0)
h = torch.randn(1, 8, 1023, 1023, device="cuda")
plan = hn.Plan((512, 512), 1, 8)
times = []
for _ in range(2):
    torch.cuda.synchronize()
    t = time.perf_counter()
    plan.forward(q, k, v, h)
    torch.cuda.synchronize()
    times.append(time.perf_counter() - t)
print("ms", (times[0] - times[1]) * 1e3)
"""


@pytest.mark.gpu
def test_first_forward_loads_its_kernels_quickly():
    """Row, core and row-back kernels of two source files: a few ms; 24 where their images were stored compressed for size (the
    best of three processes, as the first one also brings the library's file into memory)."""
    if os.environ.get("HYENAND_LIB") == "debug":
        pytest.skip("the checked build is stored compressed")
    best = 1e9
    for _ in range(3):
        r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=600)
        assert r.returncode == 0, r.stderr[-2000:]
        best = min(best, float(r.stdout.split()[-1]))
    assert best < 12, best
