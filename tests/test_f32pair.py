"""The paired FP64 -> (hi, lo) float conversion (csrc/f32conv.h) gives the bits of the two
separate conversions: random bit patterns, the fast path's exponent limits, ties, zeros."""
import ctypes
import os
import shutil
import subprocess
import tempfile

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1510_03110_gb300", "csrc")

SHIM = r'''
#include "f32conv.h"
extern "C" void pair(const double* x, float* h, float* l, float* h2, float* l2, long n)
{
    for (long i = 0; i < n; ++i) {
        mhe::f32_pair(x[i], h[i], l[i]);
        h2[i] = mhe::f32_rn(x[i]);
        l2[i] = mhe::f32_lo(x[i], h2[i]);
    }
}
'''


def test_pair_equals_the_two_conversions():
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    with tempfile.TemporaryDirectory() as d:
        src, so = os.path.join(d, "s.cpp"), os.path.join(d, "s.so")
        open(src, "w").write(SHIM)
        subprocess.run([cxx, "-O2", "-shared", "-fPIC", "-I", CSRC, src, "-o", so], check=True)
        L = ctypes.CDLL(so)
        rng = np.random.default_rng(5)
        bits = rng.integers(0, 2 ** 63, size=300000, dtype=np.uint64) * np.uint64(2) + rng.integers(0, 2, 300000, dtype=np.uint64)
        frac = bits & np.uint64(0x800FFFFFFFFFFFFF)
        edge = frac | (rng.integers(890, 1160, size=bits.size).astype(np.uint64) << np.uint64(52))   # the fast path and around
        tie = (edge & ~np.uint64(0x1FFFFFFF)) | np.uint64(0x10000000)
        x = np.concatenate([bits, edge, tie, edge & ~np.uint64(0x1FFFFFFF)]).view(np.float64)
        x = np.concatenate([x, [0.0, -0.0, 1.0, -1.0, np.inf, -np.inf, 5e-324, 3.5e38, -1e-310]])
        out = [np.empty(x.size, np.float32) for _ in range(4)]
        p = lambda a: ctypes.c_void_p(a.ctypes.data)  # noqa: E731
        L.pair(p(x), *(p(a) for a in out), ctypes.c_long(x.size))
        for a, b in ((out[0], out[2]), (out[1], out[3])):
            nan = np.isnan(a) & np.isnan(b)
            # an exact value's rest may be +0 or -0
            assert np.all((a.view(np.uint32) == b.view(np.uint32)) | nan | ((a == 0) & (b == 0)))
