"""The double-precision walk's logarithm, root, cosine and sine in 64-bit
integers (mcg_fixed.cuh, compiled for the host) against 60-digit values.

Bounds, relative, are those of the functions they stand for, where the results
are small as well (u1 next to 1, angles next to an axis): a logarithm within 1
unit in the last place, whose root, rounded, is within 2^-53 + 2^-53; cosine and
sine within 2 units, 2^-51, of those of the angle rounded to a double.  (The
hardware's reciprocal root is only a first guess; on the GPU the normals are
compared in test_gpu_edges.py.)"""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

from paper_1709_07469_gb300 import build as B

mpmath = pytest.importorskip("mpmath")

SOURCE = """
#include "mcg_fixed.cuh"
static constexpr mcg::fx::Tables T{};
extern "C" void polar(const uint32_t* w1, const uint32_t* w2, int64_t n, double* r, double* c, double* s)
{
    for (int64_t i = 0; i < n; ++i) {
        float rf;
        int64_t co, si;
        mcg::fx::polar64(T, w1[i], w2[i], r[i], rf, co, si, c[i], s[i]);
        r[i] *= 0x1p63;
        c[i] *= 0x1p-63;
        s[i] *= 0x1p-63;
    }
}
"""


@pytest.fixture(scope="module")
def polar(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed")
    src, lib = os.path.join(d, "polar.cu"), os.path.join(d, "polar.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([B.nvcc(), *B.ARCH, "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I" + B.CSRC, src, "-o",
                    lib], check=True, capture_output=True)
    fn = ctypes.CDLL(lib).polar

    def run(w1, w2):
        w1, w2 = (np.ascontiguousarray(w, dtype=np.uint32) for w in (w1, w2))
        out = np.empty((3, w1.size))
        fn(w1.ctypes.data_as(ctypes.c_void_p), w2.ctypes.data_as(ctypes.c_void_p), ctypes.c_int64(w1.size),
           *[ctypes.c_void_p(row.ctypes.data) for row in out])
        return out

    return run


def around(center, n=400):
    """Words at and near `center`, at distances of every size, and at both sides
    of the borders of the special zones."""
    rng = np.random.default_rng(center % 1000)
    d = np.concatenate([np.arange(40), np.exp2(rng.uniform(0, 24, n)).astype(np.int64),
                        (1 << 20) + np.arange(-20, 20), (1 << 23) + np.arange(-20, 20)])
    return ((center + np.concatenate([d, -d - 1])) % (1 << 32)).astype(np.uint32)


def test_radius(polar):
    w = np.concatenate([around(0), around(1 << 31), np.random.default_rng(1).integers(0, 1 << 32, 1000)])
    r = polar(w, w)[0]
    with mpmath.workdps(60):
        for a, v in zip(w, r):
            want = mpmath.sqrt(-2 * mpmath.log((int(a) + mpmath.mpf(1) / 2) / 2**32))
            assert abs(mpmath.mpf(float(v)) - want) <= want * 2.0**-52, hex(int(a))


@pytest.mark.parametrize("axis", range(4))
def test_cosine_and_sine(polar, axis):
    w = np.concatenate([around(axis << 30), np.random.default_rng(axis).integers(0, 1 << 32, 300)])
    _, c, s = polar(w, w)
    with mpmath.workdps(60):
        for a, x, y in zip(w, c, s):
            angle = mpmath.mpf(2.0 * math.pi * ((float(a) + 0.5) * 2.0**-32))
            for got, want in ((x, mpmath.cos(angle)), (y, mpmath.sin(angle))):
                assert abs(mpmath.mpf(float(got)) - want) <= abs(want) * 2.0**-51, hex(int(a))
