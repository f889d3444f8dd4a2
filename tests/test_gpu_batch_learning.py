"""What a small batch of long rows teaches the pool sizing must not make a
large batch overflow its pools and run its phases twice (in a fresh process: the
records are the process's)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = """
import ctypes, sys
sys.path.insert(0, {root!r})
import torch
import paper_2208_05683_gb300 as psf, synthetic as syn
dev = lambda t: psf.DeviceCSR.from_host(*t)
small = [dev(syn.banded_random(300, 40, k, 2.0)) for k in range(2)]
large = [dev(syn.banded_random(30000, 20, k, 2.0)) for k in range(2)]
def launches(Zs):
    s = [psf.Series(syn.coeffs("exp"), 1e-8) for _ in Zs]
    a, b = ctypes.c_int64(), ctypes.c_int64()
    psf.lib().psf_launch_count(ctypes.byref(a))
    psf.eval_batch(s, Zs)
    torch.cuda.synchronize()
    psf.lib().psf_launch_count(ctypes.byref(b))
    return b.value - a.value
for _ in range(2):
    launches(small)
print("launches", launches(large), launches(large))
"""


def test_a_large_batch_after_a_small_one_runs_once():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    p = subprocess.run([sys.executable, "-c", CHILD.format(root=root)], capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stderr[-2000:]
    first, second = map(int, p.stdout.split("launches")[1].split())
    assert first == second
