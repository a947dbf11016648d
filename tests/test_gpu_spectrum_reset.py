"""A reconstruction after a device reset leaves memory that others have been given since alone:
the thread's kept buffer is gone with the reset, and its address may be theirs."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDART = "/usr/local/cuda/lib64/libcudart.so"

CHILD = """
import ctypes, sys
import numpy as np
sys.path.insert(0, {root!r})
from paper_2506_07430_gb300 import spectrum
rt = ctypes.CDLL({cudart!r})
mu = np.random.default_rng(0).standard_normal(300) / (1 + np.arange(300))
first = spectrum(mu, 3.0, 0.5, 256)
assert rt.cudaDeviceReset() == 0
blocks = []
for size in [2 << 20] * 16 + [8192] * 64:
    p = ctypes.c_void_p()
    assert rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(size)) == 0
    assert rt.cudaMemset(p, 0x5a, ctypes.c_size_t(size)) == 0
    blocks.append((p, size))
assert rt.cudaDeviceSynchronize() == 0
for _ in range(2):
    again = spectrum(mu, 3.0, 0.5, 256)
    assert np.array_equal(first[0], again[0]) and np.array_equal(first[1], again[1])
for p, size in blocks:
    h = np.zeros(size, np.uint8)
    assert rt.cudaMemcpy(ctypes.c_void_p(h.ctypes.data), p, ctypes.c_size_t(size), 2) == 0
    assert (h == 0x5a).all(), hex(p.value)
    assert rt.cudaFree(p) == 0
"""


@pytest.mark.skipif(not os.path.exists(CUDART), reason="no shared CUDA runtime")
def test_spectrum_after_reset_leaves_other_memory_alone():
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT, cudart=CUDART)],
                       capture_output=True, text=True, timeout=200)
    assert r.returncode == 0, r.stderr[-2000:]
