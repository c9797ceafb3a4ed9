"""The library keeps nothing of a CUDA context that a reset of the device takes away: attributes of its kernels, addresses
of its variables, its memory pool.  In a process of its own, on plain driver memory: torch does not live through a reset."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import ctypes, sys
import numpy as np
from cuda.bindings import runtime as rt
from paper_2607_27744_b200 import binding

L = binding.lib()


def dev(a):
    e, p = rt.cudaMalloc(a.nbytes)
    assert e == 0 and rt.cudaMemcpy(p, a.ctypes.data, a.nbytes, rt.cudaMemcpyKind.cudaMemcpyHostToDevice)[0] == 0
    return p


def back(p, shape):
    out = np.empty(shape, np.uint16)
    assert rt.cudaMemcpy(out.ctypes.data, p, out.nbytes, rt.cudaMemcpyKind.cudaMemcpyDeviceToHost)[0] == 0
    return (out.astype(np.uint32) << 16).view(np.float32)


def bits(x):
    return (x.astype(np.float32).view(np.uint32) >> 16).astype(np.uint16)


def score():
    # whole numbers that bf16 holds: a split layer with a table of its requests, and a plain one, by kernels that ask for
    # more shared memory than a block has without asking
    g = np.random.default_rng(0)
    N, R, K, M = 20000, 50, 128, 512
    co = np.linspace(0, N, R + 1).astype(np.int32)
    XR, XC, W = g.integers(-1, 2, (R, 64)), g.integers(-1, 2, (N, K)), g.integers(-1, 2, (M, 64 + K)) * (g.random((M, 64 + K)) < 0.1)
    want = np.repeat(XR @ W[:, :64].T, np.diff(co), 0) + XC @ W[:, 64:].T
    assert np.abs(want).max() <= 256
    plan = ctypes.c_void_p()
    cod, xr, xc, w, y = dev(co), dev(bits(XR)), dev(bits(XC)), dev(bits(W)), dev(np.zeros((N, M), np.uint16))
    assert L.rocs_plan_create(ctypes.byref(plan), R, N, cod, co.ctypes.data, None) == 0
    need = L.rocs_ikbo_linear_workspace(plan, M)
    ws = dev(np.zeros(need, np.uint8))
    assert L.rocs_ikbo_linear(plan, 0, 64, K, M, xr, 64, xc, K, w, 64 + K, w + 128, 64 + K, None, 0, y, M, ws, need, None) == 0
    assert np.array_equal(back(y, (N, M)), want)
    assert L.rocs_plan_destroy(plan) == 0
    assert L.rocs_ikbo_linear_static(0, R, N, cod, 64, K, M, xr, 64, xc, K, w, 64 + K, w + 128, 64 + K, None, 0, y, M, None) == 0
    assert np.array_equal(back(y, (N, M)), want)
    detail = ctypes.c_uint32(0)
    assert L.rocs_last_device_status(ctypes.byref(detail)) == 0


score()
for _ in range(2):
    assert rt.cudaDeviceReset()[0] == 0
    score()
print("scored")
"""


def test_calls_after_a_device_reset():
    done = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert done.returncode == 0 and done.stdout.strip() == "scored", done.stdout + done.stderr
