"""What a small batch teaches the pool sizing (its launches reserve a whole
arena per warp) must not make a large one allocate tens of GB: a batch of 64
rows, then one of 16 x 20000, in a fresh process (the records are the
process's), with the device memory pool's high-water mark read after it.  The
large batch's rows of at most a few hundred entries per stage need about 5 GB
at 28 bytes an entry; 24 GB is the bound, 60 GB the pool's own limit."""
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
s = psf.Series(syn.coeffs("exp"), 1e-8)
small = [dev(syn.laplacian_1d(33)), dev(syn.scale(syn.laplacian_2d(6), 0.25))]
large = [dev(syn.laplacian_1d(20000)) for _ in range(15)] + [dev(syn.scale(syn.laplacian_2d(40), 0.25))]
cu = ctypes.CDLL("libcuda.so.1")
torch.cuda.synchronize()
d, pool, v = ctypes.c_int(), ctypes.c_void_p(), ctypes.c_uint64(0)
assert cu.cuCtxGetDevice(ctypes.byref(d)) == 0
assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), d) == 0
for _ in range(3):
    psf.eval_batch([s] * 2, small)
torch.cuda.synchronize()
HIGH = 8
assert cu.cuMemPoolSetAttribute(pool, HIGH, ctypes.byref(v)) == 0
psf.eval_batch([s] * 16, large)
torch.cuda.synchronize()
assert cu.cuMemPoolGetAttribute(pool, HIGH, ctypes.byref(v)) == 0
print("high", v.value)
"""


def test_small_batches_do_not_inflate_large_ones():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    p = subprocess.run([sys.executable, "-c", CHILD.format(root=root)], capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stderr[-2000:]
    high = int(p.stdout.split("high")[1])
    assert 0 < high < 24 << 30, f"{high / 2**30:.1f} GB"
