// tc_digits.cuh -- digits of the operands of the tensor-core interpolation and
// spreading (nufft_tc.cu), and the sums of their products in spreading.
#pragma once
#include <cuda_runtime.h>

namespace nusht {

constexpr int ND = 5;  // digits per operand, levels of products

// x = h + l, |x| <= 1, |l| <= 2^-24 |h|, in N = 5 or 6 digits:
// x = sum_i d[i] 2^(-9 - 10 i) + O(2^-50), with six O(2^-54) (the low bits of a
// pair far below 1 are rounded on the way), with integers |d[i]| <= 512 (d[2]:
// 528, it takes the leading part of l)
template <int N>
__device__ __forceinline__ void digits(float h, float l, float d[N]) {
  constexpr float C = 12582912.0f;  // 1.5 2^23: adding and subtracting it rounds to an integer
  float x = h * 512.0f;
  d[0] = __fsub_rn(__fadd_rn(x, C), C);
  x = (x - d[0]) * 1024.0f;
  d[1] = __fsub_rn(__fadd_rn(x, C), C);
  const float r = x - d[1], L = l * 536870912.0f;  // 2^29
  d[2] = __fsub_rn(__fadd_rn(__fmaf_rn(r, 1024.0f, L), C), C);
  x = __fadd_rn(__fmaf_rn(r, 1024.0f, -d[2]), L) * 1024.0f;
  d[3] = __fsub_rn(__fadd_rn(x, C), C);
  x = (x - d[3]) * 1024.0f;
  d[4] = __fsub_rn(__fadd_rn(x, C), C);
  if (N > 5) d[5] = __fsub_rn(__fadd_rn((x - d[4]) * 1024.0f, C), C);
}

// One cell of a spreading tile: the fp32 sums s[i + j] of the products a_i b_j
// as the MMAs leave them, and the integers n[0], n[1] that take over what would
// outgrow fp32's 2^24.  A point adds at most 2^18 to level 0, 2^19 to level 1,
// 0.76 2^20 to level 2 and 1.01 2^20 to level 3, so
//  * every 16 points (tc_carry2) the multiples of 1024 in level 2, at most
//    12.8 million, pass to level 1's integer;
//  * every 32 points (tc_carry) levels 0 and 1, at most 2^23 and 2^24, become
//    integers and the multiples of 1024 in level 3 pass to level 2.
// Levels 0 to 2 are then exact for any points; level 3 loses at most a few units
// of 2^-48 in 32 points (and none below 16 million), level 4 (2^-58) is an
// fp32 sum for as long as the tile is held.
__device__ __forceinline__ float tc_over(float& s) {  // s = 1024 c + r, |r| <= 512: s becomes r; returns c + 1.5 2^23
  constexpr float C = 12582912.0f;
  const float t = __fmaf_rn(s, 0x1p-10f, C);
  s = __fmaf_rn(__fsub_rn(t, C), -1024.0f, s);
  return t;
}
__device__ __forceinline__ void tc_carry2(float& s2, int& n1) {
  n1 += __float_as_int(tc_over(s2)) - 0x4b400000;  // the bits of 1.5 2^23
}
__device__ __forceinline__ void tc_carry(float& s0, float& s1, float& s2, float& s3, int& n0, int& n1) {
  n0 += __float2int_rn(s0);
  n1 += __float2int_rn(s1);
  s0 = s1 = 0.0f;
  s2 += __fsub_rn(tc_over(s3), 12582912.0f);
}
// sum_s 2^(-18 - 10 s) level_s in units of 2^-51: 2,303 products of at most 1,
// the most a tile holds, stay below 2^63
__device__ __forceinline__ long long tc_total(int n0, int n1, float s2, float s3, float s4) {
  return ((long long)n0 << 33) + ((long long)n1 << 23) + ((long long)__float2int_rn(s2) << 13) +
         (long long)__float2int_rn(__fmaf_rn(s4, 0x1p-7f, s3 * 8.0f));
}

}  // namespace nusht
