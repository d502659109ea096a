"""The first spectral solve of a process: the code of its kernels goes to the
GPU then, so it has to be small.

Bound: 5 ms.  One kernel for the five passes (0.5 MB) takes 0.7 ms, five
kernels with a copy of the butterflies per transform (4 MB) took 14 ms; the
better of two processes is taken.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = """
import time, torch
from paper_0812_2801_gb300 import emd
emd.load()
q = torch.randn(48 ** 3, dtype=torch.float64, device="cuda")
v = torch.empty_like(q)
torch.cuda.synchronize()
t = time.perf_counter()
emd.emd_poisson_static(48, 0.3, q.data_ptr(), v.data_ptr())
torch.cuda.synchronize()
print(1e3 * (time.perf_counter() - t))
"""


def test_first_solve_of_a_process():
    ms = [float(subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, check=True,
                               capture_output=True, text=True).stdout) for _ in range(2)]
    assert min(ms) < 5.0, ms
