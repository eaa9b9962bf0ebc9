"""The library's headers compiled for the host: their arithmetic runs on the CPU, with the CUDA
intrinsics they call replaced by the same IEEE operations."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = os.environ.get("CUDA_INC", "/usr/local/cuda/include")

PRELUDE = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <cuda_runtime.h>
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
static inline float2 __fadd2_rn(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
static inline float2 __fmul2_rn(float2 a, float2 b) { return make_float2(a.x * b.x, a.y * b.y); }
static inline float2 __ffma2_rn(float2 a, float2 b, float2 c)
{
    return make_float2(std::fma(a.x, b.x, c.x), std::fma(a.y, b.y, c.y));
}
static inline unsigned __float_as_uint(float f) { unsigned u; memcpy(&u, &f, 4); return u; }
static inline double __hiloint2double(int hi, int lo)
{
    const uint64_t b = (uint64_t)(uint32_t)hi << 32 | (uint32_t)lo; double d; memcpy(&d, &b, 8); return d;
}
static inline int __double2hiint(double d) { uint64_t b; memcpy(&b, &d, 8); return (int)(b >> 32); }
template <typename T> static inline T __shfl_xor_sync(unsigned, T v, int, int = 32) { return v; }
template <typename T> static inline T __shfl_sync(unsigned, T v, int, int = 32) { return v; }
using std::fma; using std::fmax; using std::fabs; using std::sqrt;
static int rsqrt_off = 0;  // units in the last place by which rsqrt is made to miss
static inline double rsqrt(double x)
{
    double r = 1.0 / std::sqrt(x);
    for (int i = 0; i < std::abs(rsqrt_off); ++i) r = std::nextafter(r, rsqrt_off > 0 ? INFINITY : 0.0);
    return r;
}
"""


def run(tmp_path, body: str, headers=("df64.cuh",)) -> str:
    """Compile PRELUDE, the headers of csrc/ and `body` (which defines main) with g++ and return what the
    program prints."""
    gxx = shutil.which("g++")
    if not gxx or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("no host compiler or CUDA headers")
    src, exe = tmp_path / "host.cpp", tmp_path / "host"
    inc = "".join(f'#include "paper_2601_11159_gb300/csrc/{h}"\n' for h in headers)
    src.write_text(PRELUDE + inc + body)
    subprocess.check_call([gxx, "-std=c++17", "-O1", "-ffp-contract=off", "-w", "-I", ROOT, "-I", CUDA_INC,
                           str(src), "-o", str(exe)])
    return subprocess.check_output([str(exe)], text=True)
