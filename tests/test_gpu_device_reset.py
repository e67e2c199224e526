"""What the library keeps between calls (its memory pool, pinned scalars) belongs
to a context: after a device reset the next call makes its own. In a process of
its own, without torch (whose own state does not outlive a reset)."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
pytestmark = pytest.mark.gpu

CODE = """
import ctypes, glob, sys
sys.path.insert(0, {root!r})
import numpy as np
from paper_2307_16051_gb300 import nl
L, rt = nl.lib(), ctypes.CDLL(sorted(glob.glob("/usr/local/cuda/lib64/libcudart.so*"))[0])
vp, sz = ctypes.c_void_p, ctypes.c_size_t

def dev(a):
    p = vp()
    assert rt.cudaMalloc(ctypes.byref(p), sz(a.nbytes)) == 0
    assert rt.cudaMemcpy(p, vp(a.ctypes.data), sz(a.nbytes), 1) == 0
    return p.value

def host(p, n, dtype):
    a = np.empty(n, dtype)
    assert rt.cudaMemcpy(vp(a.ctypes.data), vp(p), sz(a.nbytes), 2) == 0
    return a

def once():
    N, ld = 200, 256
    x = dev(np.linspace(1.0, 1.5, N))
    F, r, fn = dev(np.zeros(N)), dev(np.zeros(N)), dev(np.zeros(1))
    assert L.nl_k_residual(N, 0.9, x, None, 0, 0.0, None, F, r, fn, None) == nl.NL_OK, nl.last_error()
    A = np.zeros((N, ld), np.float32)
    A[:, :N] = 2.0 * np.eye(N)
    b, u, g = dev(np.ones(ld, np.float32)), dev(np.zeros(ld, np.float32)), dev(np.zeros(ld, np.float32))
    Ad = dev(A)
    assert L.nl_k_gemv_residual(N, Ad, ld, b, u, g, fn, None) == nl.NL_OK, nl.last_error()
    out = [host(F, N, np.float64), host(fn, 1, np.float64)]
    # (keeps pinned memory)
    st = L.nl_linsolve16(N, Ad, ld, dev(A.astype(np.float16)), ld, dev(np.arange(N, dtype=np.int32)), b, u, 1e-4, 20, 0, 30,
                         1e-4, 10, None, None, None)
    assert st == nl.NL_OK, nl.last_error()
    assert np.array_equal(host(u, N, np.float32), np.full(N, 0.5, np.float32))
    return out

ref = once()
for _ in range(3):
    assert rt.cudaDeviceReset() == 0
    for _ in range(2):
        assert all(np.array_equal(p, q) for p, q in zip(once(), ref))
print("equal")
"""


def test_calls_after_a_device_reset():
    p = subprocess.run([sys.executable, "-c", CODE.format(root=ROOT)], capture_output=True, text=True, timeout=300)
    assert p.returncode == 0 and "equal" in p.stdout, (p.returncode, p.stdout[-500:], p.stderr[-2000:])
