"""The float-pair logarithm of an integer weight (log2pair.cuh), compiled for the host and compared with
extended precision: integer arithmetic, FP32 operations and fmaf round alike on both.

Bounds: above 2^15 a pair can do no better than the rounding of its second part, half a unit of
2^-44 for logarithms up to 31, 2^-45 at most; 2^-44.9 leaves 7 % for everything else.  An FP64
logarithm split into a pair measures 2^-44.91 at most and 2^-46.22 rms on such weights."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1104_3830_gb300", "csrc")

HARNESS = """
#include <cmath>
#include <cstring>
#include <cuda_runtime.h>
#undef __device__
#undef __forceinline__
#undef __noinline__
#define __device__
#define __noinline__
#define __forceinline__ inline
static unsigned __float_as_uint(float f) { unsigned u; memcpy(&u, &f, 4); return u; }
static float __uint_as_float(unsigned u) { float f; memcpy(&f, &u, 4); return f; }
static float __fmul_rn(float a, float b) { return a * b; }
static int __double2hiint(double d) { unsigned long long u; memcpy(&u, &d, 8); return (int)(u >> 32); }
static int __double2loint(double d) { unsigned long long u; memcpy(&u, &d, 8); return (int)u; }
static double __hiloint2double(int h, int l) {
    unsigned long long u = ((unsigned long long)(unsigned)h << 32) | (unsigned)l;
    double d;
    memcpy(&d, &u, 8);
    return d;
}
using std::max;
using std::min;
#include "log2pair.cuh"
extern "C" void weights_log2(const int* w, int n, float* hi, float* lo) {
    float4 tab[256];
    for (int j = 0; j < 256; ++j) tab[j] = sa::log2_tab_entry(j);
    for (int k = 0; k < n; ++k) {
        const float2 l = sa::wlog2(tab, w[k]);
        hi[k] = l.x;
        lo[k] = l.y;
        if (k % 4 == 3) {   // four at a time: the same numbers
            float h4[4], l4[4];
            sa::wlog2_4(tab, w + k - 3, h4, l4);
            for (int e = 0; e < 4; ++e)
                if (h4[e] != hi[k - 3 + e] || l4[e] != lo[k - 3 + e]) hi[k - 3 + e] = NAN;
        }
    }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if shutil.which("g++") is None or not os.path.isdir(inc):
        pytest.skip("no g++ or CUDA headers")
    d = tmp_path_factory.mktemp("log2pair")
    src = d / "harness.cpp"
    src.write_text(HARNESS)
    so = str(d / "harness.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-w", "-I", inc, "-I", CSRC,
                    "-I", os.path.join(ROOT, "include"), str(src), "-o", so], check=True)
    return ctypes.CDLL(so)


def _errors(lib, w):
    hi, lo = np.empty(len(w), np.float32), np.empty(len(w), np.float32)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    lib.weights_log2(p(w), len(w), p(hi), p(lo))
    return (hi.astype(np.longdouble) + lo - np.log2(w.astype(np.longdouble))).astype(np.float64)


def test_weights_above_the_int16_range(lib):
    rng = np.random.default_rng(7)
    w = np.minimum(np.floor(2.0 ** rng.uniform(15.0, 31.0, 1_000_000)), 2.0 ** 31 - 1).astype(np.int32)
    # the ends of the range, and weights whose pair is hard to round
    w = np.concatenate([w, np.arange(32768, 98304), np.arange(2 ** 31 - 65536, 2 ** 31), 2 ** np.arange(15, 31),
                        [18263941, 71320028, 17170369, 460273136, 134730888]]).astype(np.int32)
    w[::7] >>= 12   # some small neighbours, whose own logarithms are not what is bounded here
    e = _errors(lib, w)
    assert np.all(np.isfinite(e))
    e = e[w >= 32768]
    assert np.max(np.abs(e)) <= 2.0 ** -44.9
    assert np.sqrt(np.mean(e * e)) <= 2.0 ** -46.2
    assert abs(np.mean(e)) <= 2.0 ** -46.2 / np.sqrt(len(e)) * 5   # no bias
