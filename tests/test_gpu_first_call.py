"""The first call of a process: what it loads.

A stepper's translation unit is loaded as a whole at its first call.  With its code packed
and the binary64 tables in every unit that took 25 ms, in which 10^10 steps could have
been done; unpacked, and without the tables where no binary64 kernel is, it takes 1 to 5.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = r"""
import time
import torch
from paper_2206_11234_gb300 import native as nat, workloads as W

x = torch.zeros(1000, dtype=torch.float64, device="cuda")
y, z = torch.zeros_like(x), torch.empty(400, dtype=torch.float64, device="cuda")
nat.fpt_normals(11, 5, 1, 0, 100, "f64", z)  # the library's own start
torch.cuda.synchronize()
for precision in ("f32_kahan", "f32_f64acc", "f64"):
    p = nat.make_params(precision=precision, m=1.0, n_max=0.1)
    t = time.perf_counter()
    nat.fpt_simulate(p, 1000, 3.0, 2.0 ** 0.5, float("inf"), 1e-3, 0.0, 1, x, y)
    print("ms", precision, 1e3 * (time.perf_counter() - t))
"""


def test_first_calls_load_little(cuda_device):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    best = {}
    for _ in range(3):
        r = subprocess.run([sys.executable, "-c", CHILD], cwd=root, capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stdout + r.stderr
        for line in r.stdout.splitlines():
            if line.startswith("ms "):
                _, precision, ms = line.split()
                best[precision] = min(float(ms), best.get(precision, 1e9))
    assert len(best) == 3 and max(best.values()) < 10.0, best
