// tc_pack.cuh -- kernel values as packed digits, the operand format of the
// tensor-core interpolation and spreading (nufft_tc.cu).
//
// psi in [0, 1] is kept as round(psi 2^59) in six balanced base-1024 digits,
//   psi = sum_i d_i 2^(-9 - 10 i),  0 <= d_0 <= 512, -512 <= d_i <= 511 (i > 0),
// in 64 bits, the size of a float pair: four 16-bit lanes with d_0, d_1 + 512,
// d_2 + 512, d_3 + 512 in their low ten bits and the fields of d_4, d_5 (+ 512)
// split over the spare bits of lanes 0, 1 and 2, 3.  A lane pair of two taps is
// then two fp16 digits after one byte permutation, one masked OR and one
// subtraction.  The products use d_0..d_4; d_5 is for readers that want the
// value itself (tc_value).
#pragma once
#include <cuda_runtime.h>

namespace nusht {

#define TC_ZERO make_uint2(0x42000000u, 0x42000200u) /* psi = 0 */

__host__ __device__ __forceinline__ uint2 tc_pack(double psi) {
  // 512 in every field below the first makes the digits unsigned
  const long long low = 512ll * (1 + (1ll << 10) + (1ll << 20) + (1ll << 30) + (1ll << 40));
  const long long y = (long long)(psi * 0x1p59 + 0.5) + low;
  auto f = [&](int i) { return (unsigned)(y >> (10 * (5 - i))) & (i ? 1023u : 0xffffu); };
  return make_uint2(f(0) | (f(4) & 31u) << 10 | (f(1) | (f(4) >> 5) << 10) << 16,
                    f(2) | (f(5) & 31u) << 10 | (f(3) | (f(5) >> 5) << 10) << 16);
}

// psi as a float pair, within 2^-54
__device__ __forceinline__ float2 tc_value(uint2 v) {
  const unsigned m = 1023u;
  const float d0 = (float)(int)(v.x & m), d1 = (float)((int)(v.x >> 16 & m) - 512), d2 = (float)((int)(v.y & m) - 512),
              d3 = (float)((int)(v.y >> 16 & m) - 512);
  const float d4 = (float)((int)((v.x >> 10 & 31u) | (v.x >> 26) << 5) - 512);
  const float d5 = (float)((int)((v.y >> 10 & 31u) | (v.y >> 26) << 5) - 512);
  // each sum of two neighbouring digits is exact; three such sums, renormalised twice
  const float a = __fmaf_rn(d0, 0x1p-9f, d1 * 0x1p-19f), b = __fmaf_rn(d2, 0x1p-29f, d3 * 0x1p-39f),
              c = __fmaf_rn(d4, 0x1p-49f, d5 * 0x1p-59f);
  const float s = __fadd_rn(a, b), e = __fsub_rn(b, __fsub_rn(s, a));
  const float l = __fadd_rn(e, c);
  const float h = __fadd_rn(s, l);
  return make_float2(h, __fsub_rn(l, __fsub_rn(h, s)));
}

}  // namespace nusht
