"""bege_search_noalloc in whatever CUDA context is current: the device's
primary one (in which bege contexts live) and a program's own driver context,
in turn.  Each has its own copy of the library's scratch array."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import ctypes, sys
import numpy as np
sys.path[:0] = [{root!r}, {root!r} + "/tests"]
import synthetic as S
from paper_1708_01609_gb300 import binding

cuda = ctypes.CDLL("libcuda.so.1")

def check(rc):
    assert rc == 0, rc

def device(a):
    p = ctypes.c_uint64()
    check(cuda.cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(a.nbytes)))
    check(cuda.cuMemcpyHtoD_v2(p, a.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(a.nbytes)))
    return p.value

def noalloc(y, rows):
    sigma, tails = np.zeros(len(rows), np.float32), np.zeros(3 * 1024, np.int32)
    total = np.zeros(1, np.uint64)
    ps = device(sigma)
    binding.bege_search_noalloc(device(y), len(y), device(rows), rows.shape[1], 0, len(rows), 4.0,
                                ps, device(tails), 1024, device(total), 0)
    check(cuda.cuCtxSynchronize())
    check(cuda.cuMemcpyDtoH_v2(sigma.ctypes.data_as(ctypes.c_void_p), ctypes.c_uint64(ps),
                               ctypes.c_size_t(sigma.nbytes)))
    return sigma

rows = S.random_samples_bank(5, 104, 2).astype(np.float32)
strain = [S.band_limited_noise(n, 1).astype(np.float32) for n in (1 << 12, 1 << 15)]
want = []
with binding.Context(0) as ctx:
    bank = ctx.bege_define_bank_samples(rows)
    for y in strain:
        job = ctx.bege_correlate(ctx.bege_load_segment(y), bank, 0, 5, 4.0)
        want.append(ctx.bege_get_sigma(job, 5))
primary, own = ctypes.c_void_p(), ctypes.c_void_p()
check(cuda.cuCtxGetCurrent(ctypes.byref(primary)))
check(cuda.cuCtxCreate_v2(ctypes.byref(own), 0, 0))
for current in (own, primary, own):
    check(cuda.cuCtxSetCurrent(current))
    for y, w in zip(strain, want):
        assert np.array_equal(noalloc(y, rows), w)
print("same")
"""


def test_noalloc_uses_the_current_context():
    r = subprocess.run([sys.executable, "-c", PROGRAM.format(root=ROOT)], capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0 and "same" in r.stdout, r.stdout + r.stderr
