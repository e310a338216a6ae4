"""The register transforms (csrc/dft_small.cuh) compiled for the host, against the defining sums."""
import os
import subprocess

import numpy as np
import pytest

from paper_2501_13512_gb300 import build

LENGTHS = (1, 2, 4, 6, 8, 10, 12, 16)
SOURCE = r"""
#include "dft_small.cuh"
using namespace vie;
template <int H, bool FWD> static void run(const double* in, double* out) {
    double2 a[H];
    for (int i = 0; i < H; ++i) a[i] = make_double2(in[2 * i], in[2 * i + 1]);
    dft<H, FWD>(a);
    for (int i = 0; i < H; ++i) { out[2 * i] = a[i].x; out[2 * i + 1] = a[i].y; }
}
extern "C" void dft_run(int h, int fwd, const double* in, double* out) {
    switch (h) {
%s
    }
}
""" % "\n".join(f"        case {h}: fwd ? run<{h}, true>(in, out) : run<{h}, false>(in, out); break;" for h in LENGTHS)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    import ctypes
    d = tmp_path_factory.mktemp("dft")
    src, so = d / "dft.cu", d / "libdft.so"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc_path(), "-std=c++17", "-O1", "-Xcompiler", "-fPIC", "-shared", "-I", build.CSRC, "-I",
                    os.path.join(build.ROOT, "include"), "-o", str(so), str(src)], check=True)
    return ctypes.CDLL(str(so))


@pytest.mark.parametrize("h", LENGTHS)
@pytest.mark.parametrize("fwd", [1, 0])
def test_transform_is_the_dft(lib, h, fwd):
    rng = np.random.default_rng(h)
    x = rng.normal(size=h) + 1j * rng.normal(size=h)
    out = np.empty(h, np.complex128)
    lib.dft_run(h, fwd, x.ctypes.data_as(__import__("ctypes").c_void_p), out.ctypes.data_as(__import__("ctypes").c_void_p))
    ref = np.fft.fft(x) if fwd else np.fft.ifft(x) * h
    # at most 7 additions and 2 products deep: 16 units of 2^-53 of the norm
    assert np.linalg.norm(out - ref) <= 16 * 2.0 ** -53 * np.linalg.norm(ref)
