"""Calls that take scratch from the pool go on after cudaDeviceReset (in a child
process: the reset ends its context)."""
import glob
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHILD = """
import ctypes as C, sys
import numpy as np
import paper_2212_04415_gb300 as pd
import pd_workloads as W
rt = C.CDLL(sys.argv[1])
L, g = pd.lib(), W.bar().grid
G, n = pd.grid_struct(g), g.n_nodes


def device(a):
    p = C.c_void_p()
    assert rt.cudaMalloc(C.byref(p), C.c_size_t(a.nbytes)) == 0
    assert rt.cudaMemcpy(p, C.c_void_p(a.ctypes.data), C.c_size_t(a.nbytes), 1) == 0
    return p


def host(p, a):
    assert rt.cudaMemcpy(C.c_void_p(a.ctypes.data), p, C.c_size_t(a.nbytes), 2) == 0
    return a


def once():
    row, col, nb = np.zeros(n + 1, np.int32), np.zeros(400000, np.int32), C.c_int64(0)
    drow, dcol = device(row), device(col)
    assert L.pd_build_neighbours(C.byref(G), drow, dcol, col.size, C.byref(nb), None) == 0
    q, u = np.random.default_rng(1).standard_normal(3000), np.linspace(0.0, 1.0, 50)
    dq, du, dout = device(q), device(u), device(np.zeros(50))
    assert L.pd_ml_inverse_cdf(1, (C.c_int64 * 1)(3000), dq, None, 50, du, dout, None) == 0
    return nb.value, host(drow, row).copy(), host(dcol, col)[: nb.value].copy(), host(dout, np.zeros(50))


first = once()
for _ in range(2):
    assert rt.cudaDeviceReset() == 0
    again = once()
    assert again[0] == first[0] and all(np.array_equal(a, b) for a, b in zip(again[1:], first[1:]))
print("same after reset")
"""


def test_pooled_calls_after_a_device_reset(built_lib):
    found = sorted(glob.glob("/usr/local/cuda/lib64/libcudart.so*"))
    if not found:
        pytest.skip("no shared CUDA runtime")
    r = subprocess.run([sys.executable, "-c", CHILD, found[0]], cwd=ROOT, env=dict(os.environ, PYTHONPATH=ROOT),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "same after reset" in r.stdout, r.stderr[-2000:]
