"""The scratch that mpdo_gemm_tc keeps between calls: bounded, given back by mpdo_destroy,
and gone with its context: after cudaDeviceReset the next product takes a new one.  A
process of its own, through the C ABI alone (a reset ends every context of a process)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

SCRIPT = r'''
import ctypes, sys
import numpy as np
rt, lib, P = ctypes.CDLL(sys.argv[1]), ctypes.CDLL(sys.argv[2]), ctypes.c_void_p

def dev(a):
    p = P()
    assert rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(a.nbytes)) == 0
    assert rt.cudaMemcpy(p, a.ctypes.data_as(P), ctypes.c_size_t(a.nbytes), 1) == 0
    return p

def free_mb():
    f, t = ctypes.c_size_t(), ctypes.c_size_t()
    assert rt.cudaMemGetInfo(ctypes.byref(f), ctypes.byref(t)) == 0
    return f.value / 2 ** 20

def product(m, n, k, seed):
    r = np.random.default_rng(seed)
    a, b, c = r.standard_normal((m, k)), r.standard_normal((k, n)), np.zeros((m, n))
    d = [dev(x) for x in (a, b, c)]
    assert lib.mpdo_gemm_tc(m, n, k, d[0], k, d[1], n, d[2], n, 1, P(None)) == 0
    assert rt.cudaMemcpy(c.ctypes.data_as(P), d[2], ctypes.c_size_t(c.nbytes), 2) == 0
    for p in d:
        rt.cudaFree(p)
    # 2^-46 of the row and column maxima (at most 6 each here) per term
    assert np.abs(c - a @ b).max() <= 2.0 ** -46 * 36 * k

product(64, 64, 64, 0)      # modules loaded
before = free_mb()
product(3000, 3100, 2000, 1)
assert before - free_mb() <= 320
lib.mpdo_destroy(P(None))
assert before - free_mb() <= 4
product(500, 400, 300, 2)
assert rt.cudaDeviceReset() == 0
product(500, 400, 300, 3)
product(64, 64, 64, 4)
print("done")
'''


def test_given_back_and_renewed():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_05871_gb300 import build as B
    lib = B.build()
    home = [os.path.join(os.path.dirname(os.path.dirname(B.NVCC)), d, "libcudart.so") for d in ("lib64", "lib")]
    rt = next((p for p in home if os.path.exists(p)), None)
    if rt is None:
        pytest.skip("no libcudart.so beside nvcc")
    r = subprocess.run([sys.executable, "-c", SCRIPT, rt, lib], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "done" in r.stdout, r.stdout + r.stderr
