"""The first execution of a plan loads no kernels: that is done with the plan."""

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FIRST = """
import time, torch
import paper_1302_6189_gb300 as md
x = torch.randn((64, 60, 40), dtype=torch.complex64, device="cuda")
y = torch.empty_like(x)
plan = md.Plan((64, 60, 40), 16)
torch.cuda.synchronize()
t = time.perf_counter()
plan.exec(x, y)
torch.cuda.synchronize()
print((time.perf_counter() - t) * 1e6)
"""


def test_the_first_execution_in_a_process():
    us = [float(subprocess.run([sys.executable, "-c", FIRST], cwd=ROOT, capture_output=True, text=True, check=True,
                               timeout=300).stdout.split()[-1]) for _ in range(3)]
    # (114 us with loaded kernels, 780 us where three are loaded on the way)
    assert min(us) <= 350, us
