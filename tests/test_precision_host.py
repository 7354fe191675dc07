"""The kernels' sums in pieces of FP32, compiled for the host from the CUDA source, against exact arithmetic."""
import ctypes
import os
import re
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1609_06634_gb300", "csrc")


def _function(source: str, name: str) -> str:
    """The text of one __device__ __forceinline__ function."""
    txt = open(os.path.join(CSRC, source)).read()
    m = re.search(r"__device__ __forceinline__ \w+ %s\(.*?\n}\n" % name, txt, flags=re.S)
    assert m, name
    return m.group(0).replace("__device__ __forceinline__", "static inline")


def _library(tmp_path, body: str):
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    src = os.path.join(tmp_path, "host.cpp")
    with open(src, "w") as f:
        f.write("#include <cmath>\n#include <cstdint>\n#include <cstring>\nusing std::fma;\n" + body)
    lib = os.path.join(tmp_path, "host.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", src, "-o", lib], check=True)
    return ctypes.CDLL(lib)


def test_squares_are_summed_beyond_float64(tmp_path):
    """A thread's share of a spectrum (33 coefficients, values falling over six decades) as squares with weights 1
    and 2: the three parts hold the sum to 2^-60, where float64's own rounding is 2^-53.  (Each square's
    error and each sum's is kept but for the last part's rounding: 66 x 2^-24 of 2^-48.)"""
    lib = _library(str(tmp_path), _function("prep_project.cu", "two_sum") + _function("prep_project.cu", "add_square") + '''
extern "C" void sum_squares(const float* x, const float* w, int n, float* out) {
    float hi = 0.f, mid = 0.f, lo = 0.f;
    for (int i = 0; i < n; ++i) add_square(hi, mid, lo, x[i], w[i]);
    out[0] = hi; out[1] = mid; out[2] = lo;
}
''')
    rng = np.random.default_rng(3)
    ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    for _ in range(200):
        x = (rng.standard_normal(66) * 10.0 ** rng.uniform(-6, 0, 66)).astype(np.float32)
        w = rng.integers(1, 3, 66).astype(np.float32)
        out = np.empty(3, dtype=np.float32)
        lib.sum_squares(ptr(x), ptr(w), 66, ptr(out))
        exact = sum(Fraction(float(b)) * Fraction(float(a)) ** 2 for a, b in zip(x, w))
        got = sum(Fraction(float(v)) for v in out)
        assert abs(got - exact) <= exact / 2 ** 60
