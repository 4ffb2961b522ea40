"""Host checks of the operand arithmetic of the tensor-core interpolation and
spreading (csrc/nufft_tc.cu): the device headers it is written in, compiled
here with g++ (the few CUDA intrinsics they use are given as plain C++).

* scaling: oz_scale(v, k) is v 2^k exactly, or 0 where that (or v) is below
  the normal range, for every exponent of v and every shift;
* scaling and split: for every exponent of a largest value and every exponent
  of a value up to it, the float pair is the scaled value within 2^-48 of it,
  and 0 below 2^-74 of the largest;
* sums: one cell of a spreading tile over up to as many points as a tile may
  hold (2,303), with fp32 accumulators that round or truncate, for operands
  whose digits all have one sign and the largest magnitude, equal operands and
  random ones.  Against the exact sum of the kept digit products the total is
  off by at most 16 units of 2^-48 per 32 points (level 3, four MMAs per 16
  points, each losing less than two units above 2^24) and two units of the
  last conversion.  Against the sum of the operands' products each point may
  lose 2^-47 (the dropped products and digits) or, with level 5 and six digits
  of one operand, 2^-50 of the other's missing digit and 2^-54 of its own.
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
struct uint2 { unsigned x, y; };
inline uint2 make_uint2(unsigned x, unsigned y) { return {x, y}; }
#define __host__
#define __forceinline__ inline
struct float2 { float x, y; };
inline float2 make_float2(float x, float y) { return {x, y}; }
template <class T, class F>
inline T bits_as(F v) {
  static_assert(sizeof(T) == sizeof(F), "");
  T r;
  std::memcpy(&r, &v, sizeof r);
  return r;
}
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

SUMS = r"""
#include <algorithm>
#include <cstdio>
#include <random>
#include "dfloat.cuh"
#include "tc_digits.cuh"
#include "tc_pack.cuh"
using namespace nusht;
typedef __int128 big;

// an fp32 accumulator after the exact sum x
static float acc32(double x, bool truncate) {
  const float f = (float)x;
  return truncate && std::fabs((double)f) > std::fabs(x) ? std::nextafterf(f, 0.0f) : f;
}
static void digits_of_psi(double psi, int d[5]) {
  const uint2 v = tc_pack(psi);
  d[0] = v.x & 1023;
  d[1] = (int)(v.x >> 16 & 1023) - 512;
  d[2] = (int)(v.y & 1023) - 512;
  d[3] = (int)(v.y >> 16 & 1023) - 512;
  d[4] = (int)((v.x >> 10 & 31) | (v.x >> 26) << 5) - 512;
}

int main() {
  std::mt19937_64 g(5);
  std::uniform_real_distribution<double> U(0.0, 1.0);
  const double top = 511 * 0x1p-9 + 511 * 0x1p-19 + 511 * 0x1p-29 + 511 * 0x1p-39 + 511 * 0x1p-49;
  long bad = 0;
  for (int n : {1, 16, 31, 256, 672, 2303})
    for (int kind = 0; kind < 20; ++kind)
      for (int truncate = 0; truncate < 2; ++truncate)
        for (int fine = 0; fine < 2; ++fine) {
          const double x0 = kind == 0 ? top : U(g), p0 = kind == 0 ? top : U(g);
          float s[ND] = {};
          int n0 = 0, n1 = 0;
          big kept = 0;  // in units of 2^-68
          long double all = 0;
          for (int q0 = 0; q0 < n; q0 += 32) {
            for (int k0 = q0; k0 < std::min(n, q0 + 32); k0 += 16) {
              long long lev[ND + 1] = {};
              for (int q = k0; q < std::min(n, k0 + 16); ++q) {
                double x = kind < 14 ? x0 : (kind < 17 ? 1.0 : (g() & 1 ? 1 : -1)) * U(g), p = kind < 14 ? p0 : U(g);
                if (kind > 10 && q % 3) x *= 0x1p-20;
                float h, l, a[ND + 1] = {};
                int b[5];
                split_qr(x, h, l);
                if (fine)
                  digits<ND + 1>(h, l, a);
                else
                  digits<ND>(h, l, a);
                digits_of_psi(p, b);
                for (int i = 0; i < ND + fine; ++i)
                  for (int j = 0; j < ND && i + j < ND + fine; ++j) {
                    lev[i + j] += (long long)a[i] * b[j];
                    kept += (big)((long long)a[i] * b[j]) << (10 * (ND - i - j));
                  }
                all += ((long double)h + (long double)l) * (long double)p;
              }
              for (int k = 0; k < ND; ++k) {
                // level 5 joins level 4 times 2^-10
                const double v = (double)s[k] + (double)lev[k] + (k == ND - 1 ? (double)lev[ND] * 0x1p-10 : 0.0);
                s[k] = acc32(v, truncate);
              }
              tc_carry2(s[2], n1);
            }
            tc_carry(s[0], s[1], s[2], s[3], n0, n1);
          }
          const long long got = tc_total(n0, n1, s[2], s[3], s[4]);  // 2^-51
          const long double rounding = 0x1p-48L * (16 * ((n + 31) / 32) + 2);
          if (std::fabs((long double)(((big)got << 17) - kept)) * 0x1p-68L > rounding) ++bad;
          const long double lost = n * (fine ? 0x1p-50L + 0x1p-54L : 0x1p-47L);
          if (std::fabs((long double)got * 0x1p-51L - all) > rounding + lost) ++bad;
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


def test_sums_of_digit_products(tmp_path):
    _run(tmp_path, SUMS)
