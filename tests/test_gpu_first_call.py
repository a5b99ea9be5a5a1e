"""What the first FP32 product of a process pays for."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROBE = """
import time, torch
import paper_2105_06806_gb300 as ed
from workloads import make_model
s = ed.Sector(make_model(1, 7, U=2.0, seed=1), 4, 4)
for p, dt in (("fp64", torch.float64), ("fp32", torch.float32)):
    v = torch.ones(s.blocked_dim, dtype=dt, device="cuda")
    w = torch.zeros_like(v)
    torch.cuda.synchronize()
    t = time.perf_counter()
    ed.matvec_blocked(s, v, w, p)
    torch.cuda.synchronize()
    t = time.perf_counter() - t
print(t)
"""


def test_first_fp32_product_loads_only_its_kernels(ed):
    """A one-orbital sector's first FP32 product (4,900 elements) loads the kernels it can
    launch, not every instance of the orbital-factorised product: those alone took 11 ms
    of 13.  Best of three processes below 6 ms (1.5 ms measured)."""
    best = min(float(subprocess.run([sys.executable, "-c", PROBE], cwd=ROOT, check=True,
                                    capture_output=True, text=True).stdout.split()[-1])
               for _ in range(3))
    assert best < 6e-3
