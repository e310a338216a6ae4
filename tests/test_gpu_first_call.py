"""The first calls of a process, made on a stream that does not wait for the legacy default stream."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# The default stream is busy (about 0.2 s of complex128 products) when the first complex64 product is asked for on
# a non-blocking stream: tables that the library uploads through the default stream must be there all the same.
# Kernels are loaded ahead: loading one on its first launch would wait for the busy stream. (Without PyTorch, whose
# kernels would be loaded as well.)
FIRST_PRODUCT = """
import ctypes, os
import numpy as np
from ctypes import byref, c_void_p
from paper_2501_13512_gb300 import build, inputs, vie

rt = ctypes.CDLL(os.path.join(os.path.dirname(os.path.dirname(build.nvcc_path())), "lib64", "libcudart.so"))
lib = vie.load()

def ok(rc):
    assert rc == 0, rc

def buffer(host):
    p = c_void_p()
    ok(rt.cudaMalloc(byref(p), ctypes.c_size_t(host.nbytes)))
    ok(rt.cudaMemcpy(p, c_void_p(host.ctypes.data), ctypes.c_size_t(host.nbytes), 1))
    return p

def grid(n, mask):
    eps_r, _, x = inputs.random_case(n, seed=1)
    g, sp = vie.Grid(eps_r, 0.05), c_void_p()
    ok(lib.vie_green_spectrum(g.handle, 2 * np.pi, mask, None, byref(sp)))
    return g, sp, x

big, bsp, bx = grid((96, 96, 96), vie.C128)
bx = buffer(bx)
by = buffer(np.zeros(3 * 96**3, np.complex128))
g, sp, x = grid((40, 20, 10), vie.C64)
x = np.ascontiguousarray(x.astype(np.complex64))
xd, yd = buffer(x), buffer(np.zeros_like(x))
stream = c_void_p()
ok(rt.cudaStreamCreateWithFlags(byref(stream), 1))
ok(rt.cudaDeviceSynchronize())
for _ in range(80):
    ok(lib.vie_matvec(big.handle, bsp, vie.C128, bx, by, None))
y = []
for _ in range(2):
    ok(lib.vie_matvec(g.handle, sp, vie.C64, xd, yd, stream))
    ok(rt.cudaDeviceSynchronize())
    y.append(np.empty_like(x))
    ok(rt.cudaMemcpy(c_void_p(y[-1].ctypes.data), yd, ctypes.c_size_t(x.nbytes), 2))
assert np.isfinite(y[1]).all() and np.abs(y[1]).max() > 0
assert np.array_equal(y[0], y[1]), "the first product differs from the second"
"""


def test_first_complex64_product_on_a_non_blocking_stream():
    p = subprocess.run([sys.executable, "-c", FIRST_PRODUCT], cwd=ROOT, capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, CUDA_MODULE_LOADING="EAGER"))
    assert p.returncode == 0, p.stderr[-2000:]
