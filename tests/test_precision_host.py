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
    """A thread's share of a spectrum (33 coefficients, sizes over six decades) as squares with weights 1
    and 2: the parts hold the sum to 2^-60, where float64's own rounding is 2^-53.  (Each square's
    error and each sum's is kept but for the last part's rounding: 66 x 2^-24 of 2^-48.)  Their total in float64 is
    rounded once, but for 2^-24 of a rounding."""
    lib = _library(str(tmp_path), '''
struct float2 { float x, y; };
static float2 make_float2(float x, float y) { return float2{x, y}; }
static float2 __fadd2_rn(float2 a, float2 b) { return {a.x + b.x, a.y + b.y}; }
static float2 __fmul2_rn(float2 a, float2 b) { return {a.x * b.x, a.y * b.y}; }
static float2 __ffma2_rn(float2 a, float2 b, float2 c) { return {fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y)}; }
''' + _function("prep_project.cu", "two_sum") + _function("prep_project.cu", "add_square") +
                   _function("prep_project.cu", "square_total") + '''
extern "C" double sum_squares(const float* x, const float* w, int n, float* out) {
    float2 hi{0.f, 0.f}, mid = hi, lo = hi;
    for (int i = 0; i < n; ++i) add_square(hi, mid, lo, float2{x[2 * i], x[2 * i + 1]}, float2{w[i], w[i]});
    const float2 r[3] = {hi, mid, lo};
    for (int k = 0; k < 3; ++k) { out[2 * k] = r[k].x; out[2 * k + 1] = r[k].y; }
    return square_total(hi, mid, lo);
}
''')
    lib.sum_squares.restype = ctypes.c_double
    rng = np.random.default_rng(3)
    ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    for _ in range(200):
        x = (rng.standard_normal(66) * 10.0 ** np.repeat(rng.uniform(-6, 0, 33), 2)).astype(np.float32)
        w = rng.integers(1, 3, 33).astype(np.float32)
        out = np.empty(6, dtype=np.float32)
        total = lib.sum_squares(ptr(x), ptr(w), 33, ptr(out))
        exact = sum(Fraction(float(b)) * Fraction(float(a)) ** 2 for a, b in zip(x, np.repeat(w, 2)))
        got = sum(Fraction(float(v)) for v in out)
        assert abs(got - exact) <= exact / 2 ** 60
        assert abs(Fraction(total) - exact) <= exact * Fraction(101, 100) / 2 ** 53


def test_exponential_of_the_reductions(tmp_path):
    """exp_neg over [-100, 0] against long double where that is wider, within 2.7e-16: half an ulp (2^-53) each of the
    table's entry and of the last sum, and the series' truncation."""
    if np.finfo(np.longdouble).nmant <= 52:
        pytest.skip("no wider type")
    lib = _library(str(tmp_path), '''
static int __double2loint(double x) { int64_t b; memcpy(&b, &x, 8); return (int)(uint32_t)b; }
static int __double2hiint(double x) { int64_t b; memcpy(&b, &x, 8); return (int)(b >> 32); }
static double __hiloint2double(int h, int l) {
    const int64_t b = (int64_t)((uint64_t)(uint32_t)h << 32 | (uint32_t)l); double x; memcpy(&x, &b, 8); return x;
}
static const int kExpBits = 8;
''' + _function("score.cu", "exp_neg") + '''
extern "C" void exps(const double* x, int n, double* y) {
    double tab[256];
    for (int j = 0; j < 256; ++j) tab[j] = exp2(j / 256.0);
    for (int i = 0; i < n; ++i) y[i] = exp_neg(x[i], tab);
}
''')
    rng = np.random.default_rng(4)
    x = np.concatenate([-rng.uniform(0, 100, 200_000), -rng.uniform(0, 1, 50_000), [0.0, -100.0, -1e-300, -np.log(2.0)]])
    y = np.empty_like(x)
    lib.exps(x.ctypes.data_as(ctypes.c_void_p), len(x), y.ctypes.data_as(ctypes.c_void_p))
    exact = np.exp(x.astype(np.longdouble))
    assert float(np.abs((y - exact) / exact).max()) < 2.7e-16
