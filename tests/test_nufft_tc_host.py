"""Host checks of the operand arithmetic of the tensor-core interpolation and
spreading (csrc/nufft_tc.cu): the device headers it is written in, compiled
here with g++ (the few CUDA intrinsics they use are given as plain C++).

* scaling: oz_scale(v, k) is v 2^k exactly, or 0 where that (or v) is below
  the normal range, for every exponent of v and every shift;
* scaling and split: for every exponent of a largest value and every exponent
  of a value up to it, the float pair is the scaled value within 2^-48 of it,
  and 0 below 2^-74 of the largest.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2406_14542_gb300", "csrc")

INTRINSICS = r"""
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>
#define __device__
#define __host__
#define __forceinline__ inline
struct float2 { float x, y; };
inline float2 make_float2(float x, float y) { return {x, y}; }
template <class T, class F> inline T bits_as(F v) { T r; static_assert(sizeof(T) == sizeof(F), ""); std::memcpy(&r, &v, sizeof r); return r; }
inline int __double2hiint(double v) { return (int)(bits_as<uint64_t>(v) >> 32); }
inline int __double2loint(double v) { return (int)(uint32_t)bits_as<uint64_t>(v); }
inline float __uint_as_float(unsigned v) { return bits_as<float>(v); }
inline unsigned __float_as_uint(float v) { return bits_as<unsigned>(v); }
inline float __int_as_float(int v) { return bits_as<float>(v); }
inline int __float_as_int(float v) { return bits_as<int>(v); }
inline float __int2float_rn(int v) { return (float)v; }
inline float __uint2float_rn(unsigned v) { return (float)v; }
inline float __double2float_rn(double v) { return (float)v; }
inline int __float2int_rn(float v) { return (int)std::lrintf(v); }
inline unsigned __funnelshift_l(unsigned lo, unsigned hi, int s) { return (hi << s) | (lo >> (32 - s)); }
inline float __fadd_rn(float a, float b) { return a + b; }
inline float __fsub_rn(float a, float b) { return a - b; }
inline float __fmul_rn(float a, float b) { return a * b; }
inline float __fmaf_rn(float a, float b, float c) { return std::fmaf(a, b, c); }
"""

SCALE = r"""
#include <cfloat>
#include <cstdio>
#include "dfloat.cuh"
#include "ozsplit.cuh"
using namespace nusht;

int main() {
  long bad = 0;
  const double mant[] = {1.0, 1.0 + DBL_EPSILON, 1.5, 2.0 - DBL_EPSILON, 1.2345678901234567, -1.0, -1.9999999999};
  for (int ex = -1074; ex <= 1023; ++ex)
    for (int k = -2100; k <= 2100; ++k) {
      if (ex + k > 1022) break;
      for (double f : mant) {
        const double v = std::ldexp(f, ex);
        const bool normal = std::isnormal(v) && std::ilogb(v) + k >= -1022;
        if (oz_scale(v, k) != (normal ? std::ldexp(v, k) : 0.0)) ++bad;
      }
    }
  if (oz_scale(0.0, -500) != 0.0 || oz_scale(-0.0, 500) != 0.0) ++bad;
  // a largest value below 2^fe, values of every exponent up to it
  for (int fe = -899; fe <= 128; ++fe)
    for (int ex = -1074; ex < fe; ++ex)
      for (double f : mant) {
        const double v = std::ldexp(f, ex);
        float h, l;
        split_qr(oz_scale(v, -fe), h, l);
        const double got = (double)h + (double)l, want = std::ldexp(v, -fe);
        if (std::fabs(want) < 0x1p-74 ? got != 0.0 : !(std::fabs(got - want) <= std::fabs(want) * 0x1p-48)) ++bad;
      }
  std::printf("%ld\n", bad);
  return bad != 0;
}
"""


def _run(tmp_path, code):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    (tmp_path / "cuda_runtime.h").write_text(INTRINSICS)
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text('#include "cuda_runtime.h"\n' + code)
    subprocess.check_call([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-I", str(tmp_path), "-I", CSRC, str(src),
                           "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr


def test_scale_and_split_of_every_exponent(tmp_path):
    _run(tmp_path, SCALE)
