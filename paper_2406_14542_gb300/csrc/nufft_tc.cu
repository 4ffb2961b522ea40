// nufft_tc.cu -- interpolation and spreading of FP64 plans as exact integer
// products on the tensor cores.
//
// For the points of one 16 x 16-cell bin the taps fall into a tile of at most
// 32 x 32 fine-grid cells (w <= 17), and both steps are small dense products
// with zero-padded kernel rows:
//   interpolation  D[p][a] = sum_b psi2_p[b] U[a][b],   f_p = sum_a psi1_p[a] D[p][a];
//   spreading      U[a][b] = sum_p (f_p psi1_p[a]) psi2_p[b].
// The float-pair kernels (nufft.cu) spend 13 FP32 instructions on each of a
// point's w^2 taps; here the taps are tensor-core work and a point costs the
// splitting of its 2 w kernel values and, in interpolation, w float-pair
// multiply-adds: about 100 (interpolation) and 125 (spreading) warp instructions
// a point instead of 150 and 220 at w = 14.  At lmax 1023 (2.1M points)
// interpolation 329 -> 285 us, spreading 534 -> 378; at lmax 4095 (33.6M) 5.08
// -> 4.43 and 8.00 -> 5.69 ms.  What bounds both is issue (62 and 59 % of the
// slots) and the latency of the points' reads and of the block's phases; the
// tensor pipe is idle three quarters of the time.
//
// Exact products.  An operand scaled to |x| <= 1 is written in five balanced
// digits, x = sum_i d_i 2^(-9 - 10 i) with integers |d_i| <= 528, each exact in
// fp16.  mma.sync (fp16 operands, fp32 accumulation) forms the 15 digit
// products with i + j <= 4; the products of one level i + j accumulate into one
// fp32 sum, which holds integers exactly up to 2^24.  Interpolation adds w <= 17
// nonzero terms per product: levels 0 to 2 stay below 2^24, levels 3 and 4
// (2^-48 and 2^-58 of the scales) may round their last bit.  Spreading adds any
// number of points and moves what would outgrow 2^24 into integers
// (tc_digits.cuh).  What is dropped (level 5 on) is below 2^-48 of the operands'
// scales: the tile's largest grid value; the largest point value of a block, a
// run of up to TC_RUN subproblems; the kernel's 1.  For the widest kernels
// (FINE) level 5 is kept, its operands scaled by 2^-10 into level 4's sum, and
// the values of a spreading block, which may lie far below their scale, have a
// sixth digit.  The sum of the levels is carried as a float pair or a 64-bit
// integer.
//
// The warp-level MMA serves this shape: products of 16 points (or cells) by 8,
// operands made by the warps that consume them at once.  At its 1024
// multiply-adds per clock and SM a point takes 15 cycles of the tensor pipe,
// less than its instructions take to issue, so a faster matrix unit fed
// through descriptors and tensor memory would not shorten the step.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "dfloat.cuh"
#include "nusht_internal.cuh"
#include "ozsplit.cuh"
#include "tc_digits.cuh"
#include "tc_pack.cuh"

namespace nusht {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int BIN = 16;      // bin edge the kernels are written for
constexpr int TC_SUB = 256;  // most points of a subproblem
constexpr int GP = 16;       // points per interpolation group (rows of one MMA)
constexpr int CP = 32;       // points per spreading chunk
constexpr int ST = 256;      // threads of a spreading block
constexpr int TC_RUN = 8;    // most subproblems per spreading block

// digit matrices have rows of 32 halves, their four 16-byte chunks permuted by
// the row so that ldmatrix (eight rows of one chunk) is conflict-free
__device__ __forceinline__ int at(int row, int col) {
  return row * 32 + ((((col >> 3) ^ (row >> 1)) & 3) << 3) + (col & 7);
}

// the digits of two neighbouring columns (x even, y odd) into matrices `stride`
// halves apart, from packed kernel values (tc_pack)
__device__ __forceinline__ void put_packed(__half* dst, int stride, uint2 x, uint2 y) {
  const unsigned p0 = __byte_perm(x.x, y.x, 0x5410), p1 = __byte_perm(x.x, y.x, 0x7632);
  const unsigned p2 = __byte_perm(x.y, y.y, 0x5410), p3 = __byte_perm(x.y, y.y, 0x7632);
  // a 10-bit field under the exponent 2^10 is the fp16 number 1024 + field
  auto num = [](unsigned v, float bias) {
    const unsigned h = (v & 0x03ff03ffu) | 0x64006400u;
    return __hsub2(*reinterpret_cast<const __half2*>(&h), __float2half2_rn(bias));
  };
  auto put = [&](int i, __half2 v) { *reinterpret_cast<__half2*>(dst + i * stride) = v; };
  put(0, num(p0, 1024.f));
  put(1, num(p1, 1536.f));
  put(2, num(p2, 1536.f));
  put(3, num(p3, 1536.f));
  put(4, num(((p0 >> 10) & 0x001f001fu) | ((p1 >> 5) & 0x03e003e0u), 1536.f));
}

// ... and N digits from float pairs
template <int N>
__device__ __forceinline__ void put_pairs(__half* dst, int stride, float2 x, float2 y) {
  float dx[N], dy[N];
  digits<N>(x.x, x.y, dx);
  digits<N>(y.x, y.y, dy);
#pragma unroll
  for (int i = 0; i < N; ++i) *reinterpret_cast<__half2*>(dst + i * stride) = __floats2half2_rn(dx[i], dy[i]);
}

__device__ __forceinline__ void mma(float d[4], const unsigned a[4], unsigned b0, unsigned b1) {
  asm(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// two digits times 2^-10, still exact in fp16: their products go one level up
__device__ __forceinline__ unsigned up_level(unsigned v) {
  const __half2 h = __hmul2(*reinterpret_cast<__half2*>(&v), __float2half2_rn(0x1p-10f));
  return *reinterpret_cast<const unsigned*>(&h);
}
__device__ __forceinline__ void ldm4(unsigned r[4], const __half* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((unsigned)__cvta_generic_to_shared(p))
               : "memory");
}
__device__ __forceinline__ void ldm2(unsigned r[2], const __half* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];"
               : "=r"(r[0]), "=r"(r[1])
               : "r"((unsigned)__cvta_generic_to_shared(p))
               : "memory");
}
__device__ __forceinline__ void ldm2t(unsigned r[2], const __half* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
               : "=r"(r[0]), "=r"(r[1])
               : "r"((unsigned)__cvta_generic_to_shared(p))
               : "memory");
}
__device__ __forceinline__ void ldm4t(unsigned r[4], const __half* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((unsigned)__cvta_generic_to_shared(p))
               : "memory");
}

// s0 + 2^-10 s1 + 2^-20 s2 + 2^-30 s3 + 2^-40 s4 as a float pair
__device__ __forceinline__ float2 levels(float s0, float s1, float s2, float s3, float s4) {
  auto two_sum = [](float a, float b, float& e) {
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return s;
  };
  float e1, e2;
  float h = two_sum(s0, s1 * 0x1p-10f, e1);
  h = two_sum(h, s2 * 0x1p-20f, e2);
  return make_float2(h, __fmaf_rn(__fmaf_rn(s4, 0x1p-10f, s3), 0x1p-30f, __fadd_rn(e1, e2)));
}

// Operands are scaled by oz_scale: a value so far below the largest that its
// scaled exponent would leave the double range is zero (split_qr drops
// everything below 2^-74 of the largest in any case).
// The largest magnitude of an operand, as a double's high word without its
// sign: 2^exp_of bounds it; below 2^-900 it counts as zero, from 2^128 on (an
// infinity or NaN among them; the FFT stages' float pairs end there) the
// results are NaN
__device__ __forceinline__ int exp_of(int hi) { return (hi >> 20) - 1022; }
__device__ __forceinline__ bool too_small(int hi) { return hi < (1023 - 900) << 20; }
__device__ __forceinline__ bool too_large(int hi) { return hi >= (1023 + 128) << 20; }
__device__ __forceinline__ double quiet_nan() { return __longlong_as_double(0x7ff8000000000000ll); }

// ---------------------------------------------------------------------------
// interpolation: one block per subproblem; the tile's digits are made once, a
// warp takes 16 points at a time
// ---------------------------------------------------------------------------
struct __align__(16) InterpSmem {
  __half U[ND][32 * 32];     // U[a][b]
  __half P[4][ND][GP * 32];  // per warp: psi2 of 16 points, shifted to tile columns
  int mx[4];
};

template <bool FINE>
__global__ void __launch_bounds__(128, 7) interp_tc_k(const double* __restrict__ grid, int64_t stride, int n1, int n2,
                                                      int nb2, int w, float ipw, const int* __restrict__ sub,
                                                      const int* __restrict__ cell, const float2* __restrict__ psi,
                                                      const int* __restrict__ perm, double* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  InterpSmem& sm = *reinterpret_cast<InterpSmem*>(smem_raw);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int bin = sub[3 * blockIdx.x], start = sub[3 * blockIdx.x + 1], cnt = sub[3 * blockIdx.x + 2];
  const int r0 = (bin / nb2) * BIN, c0 = (bin % nb2) * BIN;
  const int2* cells = reinterpret_cast<const int2*>(cell) + start;
  // tile rows that some point reaches (the points are in cell order): the grid
  // holds values only in such rows (the row FFT passes leave the others as
  // they were), so the rest of the tile is zero
  const int lo = cells[0].x - r0, hi = cells[cnt - 1].x - r0 + w - 1;
  // two neighbouring columns of four rows per thread, and the largest magnitude
  const int tc = 2 * (threadIdx.x & 15), tr0 = threadIdx.x >> 4;
  double u[4][2];
  int mx = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int tr = tr0 + 8 * k;
    int r = r0 + tr;
    while (r >= n1) r -= n1;  // the halo may wrap more than once on tiny grids
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      int c = c0 + tc + e;
      while (c >= n2) c -= n2;
      u[k][e] = tr >= lo && tr <= hi && tc + e < BIN + w - 1 ? grid[(int64_t)r * stride + c] : 0.0;
      mx = max(mx, __double2hiint(u[k][e]) & 0x7fffffff);
    }
  }
  mx = __reduce_max_sync(FULL, mx);
  if (lane == 0) sm.mx[warp] = mx;
  __syncthreads();
  mx = max(max(sm.mx[0], sm.mx[1]), max(sm.mx[2], sm.mx[3]));
  if (too_large(mx)) {
    for (int q = threadIdx.x; q < cnt; q += 128) out[perm[start + q]] = quiet_nan();
    return;
  }
  const int ue = exp_of(mx);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    float2 x, y;
    split_qr(too_small(mx) ? 0.0 : oz_scale(u[k][0], -ue), x.x, x.y);
    split_qr(too_small(mx) ? 0.0 : oz_scale(u[k][1], -ue), y.x, y.y);
    put_pairs<ND>(sm.U[0] + at(tr0 + 8 * k, tc), 32 * 32, x, y);
  }
  __syncthreads();
  __half* P = sm.P[warp][0];
  const int g4 = lane >> 2, t4 = lane & 3;
  const int npw = (w + 2) >> 1;  // column pairs that hold w taps at either parity
  for (int p0 = warp * GP; p0 < cnt; p0 += 4 * GP) {
    const int np = min(GP, cnt - p0);
    const int64_t s0 = (int64_t)start + p0;
    int lr = 0, lc = 0;
    if (lane < np) {
      const int2 c = cells[p0 + lane];
      lr = c.x - r0;
      lc = c.y - c0;
    }
    // blocks of eight tile rows that some point of the group reaches
    const int glo = __shfl_sync(FULL, lr, 0), ghi = __shfl_sync(FULL, lr, np - 1) + w - 1;
    float4* z = reinterpret_cast<float4*>(P);
    for (int t = lane; t < ND * GP * 4; t += 32) z[t] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncwarp();
    for (int t0 = 0; t0 < np * npw; t0 += 64) {
      uint2 x[2], y[2];
      int o[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int t = t0 + 32 * k + lane;
        const bool in = t < np * npw;
        // p = t / npw from a float reciprocal: (t + 1/2) / npw is at least 1 / (2 npw) from an integer
        const int p = in ? __float2int_rz(((float)t + 0.5f) * ipw) : 0;
        const int pc = __shfl_sync(FULL, lc, p);
        const int b = 2 * (t - p * npw) - (pc & 1);  // taps b, b + 1 in columns pc + b (even), pc + b + 1
        const uint2* ps = reinterpret_cast<const uint2*>(psi + (s0 + p) * 2 * w + w);
        x[k] = in && b >= 0 && b < w ? __ldg(ps + b) : TC_ZERO;
        y[k] = in && b + 1 < w ? __ldg(ps + b + 1) : TC_ZERO;
        o[k] = in ? at(p, pc + b) : -1;
      }
#pragma unroll
      for (int k = 0; k < 2; ++k)
        if (o[k] >= 0) put_packed(P + o[k], GP * 32, x[k], y[k]);
    }
    __syncwarp();
    float fh[2] = {0.f, 0.f}, fl[2] = {0.f, 0.f};  // rows g4 and g4 + 8
    const int plr[2] = {__shfl_sync(FULL, lr, g4), __shfl_sync(FULL, lr, g4 + 8)};
    const int po = t4 < 2 && g4 + 8 * t4 < np ? perm[s0 + g4 + 8 * t4] : 0;  // lane t4 = 0, 1 stores row g4, g4 + 8
    for (int n0 = glo; n0 <= ghi; n0 += 8) {  // eight tile rows at a time
      float2 q[2][2];
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int p = g4 + 8 * r, a = n0 + 2 * t4 - plr[r];  // taps a, a + 1
        const float2* ps = psi + (s0 + p) * 2 * w + a;
        q[r][0] = p < np && a >= 0 && a < w ? __ldg(ps) : make_float2(0.f, 0.f);
        q[r][1] = p < np && a + 1 >= 0 && a + 1 < w ? __ldg(ps + 1) : make_float2(0.f, 0.f);
      }
      float acc[ND][4];
#pragma unroll
      for (int s = 0; s < ND; ++s)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[s][c] = 0.f;
#pragma unroll
      for (int ks = 0; ks < 2; ++ks) {
        unsigned A[ND][4];
#pragma unroll
        for (int i = 0; i < ND; ++i) ldm4(A[i], P + i * GP * 32 + at(lane & 15, ks * 16 + (lane >> 4) * 8));
#pragma unroll
        for (int j = 0; j < ND; ++j) {
          unsigned B[2];
          // rows past the tile meet psi1 = 0
          ldm2(B, sm.U[j] + at(min(n0 + (lane & 7), 31), ks * 16 + ((lane >> 3) & 1) * 8));
#pragma unroll
          for (int i = 0; i + j < ND; ++i) mma(acc[i + j], A[i], B[0], B[1]);
          if (FINE && j > 0) mma(acc[ND - 1], A[ND - j], up_level(B[0]), up_level(B[1]));
        }
      }
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const float2 x = levels(acc[0][2 * r], acc[1][2 * r], acc[2][2 * r], acc[3][2 * r], acc[4][2 * r]);
        const float2 y = levels(acc[0][2 * r + 1], acc[1][2 * r + 1], acc[2][2 * r + 1], acc[3][2 * r + 1],
                                acc[4][2 * r + 1]);
        df_mac(fh[r], fl[r], x.x, x.y, q[r][0].x, q[r][0].y);
        df_mac(fh[r], fl[r], y.x, y.y, q[r][1].x, q[r][1].y);
      }
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
#pragma unroll
      for (int o = 1; o < 4; o *= 2) {
        const float oh = __shfl_xor_sync(FULL, fh[r], o), ol = __shfl_xor_sync(FULL, fl[r], o);
        df_add(fh[r], fl[r], oh, ol);
      }
    }
    if (t4 < 2 && g4 + 8 * t4 < np)
      out[po] = oz_scale(df_value(t4 ? fh[1] : fh[0], t4 ? fl[1] : fl[0]), too_small(mx) ? 0 : ue - 18);
    __syncwarp();  // P is refilled by the next group
  }
}

// ---------------------------------------------------------------------------
// spreading: a block takes a run of consecutive subproblems (mostly bins next
// to each other along phi).  Each of the eight warps owns 16 x 8 cells of the
// tile; moving one bin on, the right half of the old tile is the left half of the
// new one, so the warps of the left half write their sums out and take the new
// right half: a cell is added to the grid twice instead of four times.  32
// points at a time are split into digits by the whole block, a pair of tile
// rows and a pair of tile columns of one point per thread.
// ---------------------------------------------------------------------------
template <int NA>
struct __align__(16) SpreadSmem {
  __half A[NA][CP * 32];             // f_p psi1_p, [point][tile row]
  __half B[ND][CP * 32];             // psi2_p, [point][tile column]
  float2 f[TC_RUN * TC_SUB];         // the run's values (scaled, as float pairs)
  unsigned char cell[TC_RUN * TC_SUB];  // and first taps, 16 (row) + column
  int sub[3 * TC_RUN];
  int mx[ST / 32];
};

template <bool FINE>
__global__ void __launch_bounds__(ST, 4) spread_tc_k(double* __restrict__ grid, int64_t stride, int n1, int n2,
                                                      int nb2, int w, float ipw, const int* __restrict__ sub, int nsub,
                                                      int run, const int* __restrict__ cell,
                                                      const float2* __restrict__ psi, const int* __restrict__ perm,
                                                      const double* __restrict__ f, float2* __restrict__ scratch) {
  constexpr int NA = FINE ? ND + 1 : ND;  // digits of f_p psi1_p
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SpreadSmem<NA>& sm = *reinterpret_cast<SpreadSmem<NA>*>(smem_raw);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i0 = blockIdx.x * run, ni = min(run, nsub - i0);
  if ((int)threadIdx.x < 3 * ni) sm.sub[threadIdx.x] = sub[3 * i0 + threadIdx.x];
  __syncthreads();
  // the run's points (contiguous) and their largest magnitude
  const int64_t start = sm.sub[1];
  const int tot = sm.sub[3 * ni - 2] + sm.sub[3 * ni - 1] - sm.sub[1];
  const int tw = BIN + w - 1;
  int mx = 0;
  for (int q = threadIdx.x; q < tot; q += ST) {
    const int2 c = reinterpret_cast<const int2*>(cell)[start + q];
    const double v = f[perm[start + q]];
    sm.cell[q] = (unsigned char)((c.x % BIN) * BIN + c.y % BIN);
    reinterpret_cast<double*>(sm.f)[q] = v;
    mx = max(mx, __double2hiint(v) & 0x7fffffff);
  }
  mx = __reduce_max_sync(FULL, mx);
  if (lane == 0) sm.mx[warp] = mx;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < ST / 32; ++k) mx = max(mx, sm.mx[k]);
  const bool bad = too_large(mx), none = bad || too_small(mx);
  const int fe = exp_of(mx);
  for (int q = threadIdx.x; q < tot; q += ST) {  // a thread's own values
    float2 v;
    split_qr(none ? 0.0 : oz_scale(reinterpret_cast<const double*>(sm.f)[q], -fe), v.x, v.y);
    sm.f[q] = v;
  }
  const int m0 = (warp >> 2) * 16;
  const int npw = (w + 2) >> 1;
  int nn0 = (warp & 3) * 8;
  int sum[2][4];
  float acc[ND][4];
  auto clear = [&]() {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      sum[0][c] = sum[1][c] = 0;
#pragma unroll
      for (int s = 0; s < ND; ++s) acc[s][c] = 0.f;
    }
  };
  // this warp's quadrant of the tile at (r0, c0) to the grid, or to the tile
  // slot of the (one) subproblem
  auto flush = [&](int r0, int c0) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int tr = m0 + (lane >> 2) + 8 * (c >> 1), tc = nn0 + 2 * (lane & 3) + (c & 1);
      if (tr >= tw || tc >= tw) continue;
      const long long v = tc_total(sum[0][c], sum[1][c], acc[2][c], acc[3][c], acc[4][c]);
      const double x = bad ? quiet_nan() : oz_dbl(v, fe - 51);
      if (scratch) {
        float2 o;
        df_of(x, o.x, o.y);
        scratch[(size_t)blockIdx.x * tw * tw + tr * tw + tc] = o;
      } else if (v != 0 || bad) {
        int r = r0 + tr, cc = c0 + tc;
        while (r >= n1) r -= n1;
        while (cc >= n2) cc -= n2;
        atomicAdd(grid + (int64_t)r * stride + cc, x);
      }
    }
    clear();
  };
  clear();
  int held = 0;  // points summed since the tile was last empty: the integers hold 2^31 / 2^19 of them
  for (int k = 0, q0 = 0; k < ni; ++k) {
    const int bin = sm.sub[3 * k], cnt = sm.sub[3 * k + 2];
    const int r0 = (bin / nb2) * BIN, c0 = (bin % nb2) * BIN;
    for (int p0 = q0; p0 < q0 + cnt; p0 += CP) {
      const int np = min(CP, q0 + cnt - p0);
      float4* z = reinterpret_cast<float4*>(sm.A[0]);
      for (int t = threadIdx.x; t < (NA + ND) * CP * 4; t += ST) z[t] = make_float4(0.f, 0.f, 0.f, 0.f);
      __syncthreads();
      for (int t = threadIdx.x; t < np * npw; t += ST) {
        const int p = __float2int_rz(((float)t + 0.5f) * ipw);  // t / npw, as in interp_tc_k
        const int cl = sm.cell[p0 + p], cr = cl >> 4, cc = cl & 15;
        const float2* ps = psi + (start + p0 + p) * 2 * w;
        const uint2* pk = reinterpret_cast<const uint2*>(ps + w);
        // taps a, a + 1 in rows cr + a (even), ... and b, b + 1 in columns cc + b
        const int i = 2 * (t - p * npw), a = i - (cr & 1), b = i - (cc & 1);
        const float2 zero = make_float2(0.f, 0.f);
        const float2 x = a >= 0 && a < w ? __ldg(ps + a) : zero, y = a + 1 < w ? __ldg(ps + a + 1) : zero;
        const uint2 xb = b >= 0 && b < w ? __ldg(pk + b) : TC_ZERO, yb = b + 1 < w ? __ldg(pk + b + 1) : TC_ZERO;
        const float2 fp = sm.f[p0 + p];
        put_packed(sm.B[0] + at(p, cc + b), CP * 32, xb, yb);
        put_pairs<NA>(sm.A[0] + at(p, cr + a), CP * 32, df_mul(x, fp), df_mul(y, fp));
      }
      __syncthreads();
      for (int ks = 0; ks * 16 < np; ++ks) {
        unsigned B[ND][2];
#pragma unroll
        for (int j = 0; j < ND; ++j)
          ldm2t(B[j], sm.B[j] + at(ks * 16 + ((lane >> 3) & 1) * 8 + (lane & 7), nn0));
#pragma unroll
        for (int i = 0; i < NA; ++i) {
          unsigned A[4];
          ldm4t(A, sm.A[i] + at(ks * 16 + (lane >> 4) * 8 + (lane & 7), m0 + ((lane >> 3) & 1) * 8));
#pragma unroll
          for (int j = 0; i + j < ND; ++j) mma(acc[i + j], A, B[j][0], B[j][1]);
          if (FINE && i > 0) mma(acc[ND - 1], A, up_level(B[ND - i][0]), up_level(B[ND - i][1]));
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) tc_carry2(acc[2][c], sum[1][c]);
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) tc_carry(acc[0][c], acc[1][c], acc[2][c], acc[3][c], sum[0][c], sum[1][c]);
      __syncthreads();  // A and B are refilled by the next chunk
    }
    q0 += cnt;
    held += cnt;
    const int next = k + 1 < ni ? sm.sub[3 * k + 3] : -1;
    if (next == bin && held < 2048) continue;
    if (next == bin + 1 && bin % nb2 + 1 < nb2 && held < 2048) {
      // one bin on: the left half is complete, the right half becomes the left
      if (nn0 < 16) flush(r0, c0);
      nn0 ^= 16;
    } else {
      flush(r0, c0);
      held = 0;
    }
  }
}

}  // namespace

// Whether the plan's interpolation and spreading run on the tensor cores: tiles
// of 32 cells (16-cell bins, w <= 17), kernels wide enough and bins full enough
// (points per subproblem, on average) for the dense products to pay.  Float
// pairs : this file, interpolation + spreading in us, uniform points, lmax 1023
// (18,400 bins):
//   points a bin      16          26          38          64
//   w = 12        248 : 293   303 : 334   369 : 376   503 : 478
//   w = 13        260 : 296   318 : 336   384 : 380   519 : 481
//   w = 14        287 : 301   352 : 339   426 : 386   584 : 492
//   w = 15        329 : 304   404 : 342   491 : 389   674 : 501
// (w = 9, 112 points: 538 : 760).  A few thousand bins do not fill the device, and
// the shorter blocks of this file hide their latency better: at lmax 383 (2,600
// bins, 16 points) w = 12 takes 61 : 56 us, w = 14 65 : 59; at lmax 511 (4,600) 80
// : 82 and 89 : 86, with 38 points 112 : 106 and 131 : 112.
constexpr int TC_WMIN = 12;
static int tc_fill(nusht_plan_t p) {
  const int w = p->sz.w;
  return p->pts.nsub <= 32 * p->sms || w > 14 ? 16 : w == 14 ? 20 : w == 13 ? 32 : 40;
}
bool nufft_tc(nusht_plan_t p) {
  const PointData& d = p->pts;
  return p->precision == NUSHT_FP64 && !p->opts.fp64_contraction && d.bin == BIN && p->sz.w >= TC_WMIN &&
         p->sz.w <= 17 && d.npts >= (int64_t)tc_fill(p) * d.nsub;
}

// Whether level 5 is kept, by the spreading kernel's own error, about
// e^(-pi w sqrt(1 - 1 / sigma)).  Without it the digits lose 2^-48 of their
// scales, which the deconvolution raises to 1e-13 of an adjoint (2.5e-13 where
// the values of a block span six decades): more than float pairs, and to be
// seen beside a kernel error below 1e-12 (w = 16 at sigma 1.5: adjoint of such a
// map, lmax 200, against 128-bit sums: float pairs 6.7e-13, without level 5
// 6.9e-13, with it 6.6e-13; w = 17: 1.30e-13, 2.77e-13, 1.31e-13).  It costs 2.1M
// points at lmax 1023, w = 17 interpolation 338 -> 360 us, spreading 439 -> 485.
constexpr double TC_FINE = 1e-12;
static bool fine_products(nusht_plan_t p) {
  return std::exp(-M_PI * p->sz.w * std::sqrt(1.0 - 1.0 / p->sz.sigma)) < TC_FINE;
}

int tc_smem_optin() {
  auto set = [](auto k, size_t n) {
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)n);
  };
  NUSHT_CUDA(set(interp_tc_k<false>, sizeof(InterpSmem)));
  NUSHT_CUDA(set(interp_tc_k<true>, sizeof(InterpSmem)));
  NUSHT_CUDA(set(spread_tc_k<false>, sizeof(SpreadSmem<ND>)));
  NUSHT_CUDA(set(spread_tc_k<true>, sizeof(SpreadSmem<ND + 1>)));
  return NUSHT_OK;
}

int tc_interp(nusht_plan_t p, double* d_map, cudaStream_t s) {
  const nusht_sizes& z = p->sz;
  auto go = [&](auto k, size_t sm) {
    k<<<p->pts.nsub, 128, sm, s>>>((const double*)p->fine, 2 * (z.n2 / 2 + 1), z.n1, z.n2, p->pts.nbins2, z.w,
                                   1.0f / (float)((z.w + 2) / 2), p->pts.sub, p->pts.cell,
                                   reinterpret_cast<const float2*>(p->pts.psi), p->pts.perm, d_map);
  };
  if (fine_products(p))
    go(interp_tc_k<true>, sizeof(InterpSmem));
  else
    go(interp_tc_k<false>, sizeof(InterpSmem));
  NUSHT_CUDA(cudaGetLastError());
  return NUSHT_OK;
}

int tc_spread(nusht_plan_t p, const double* d_map, float2* tiles, cudaStream_t s) {
  const nusht_sizes& z = p->sz;
  // runs as long as three waves of blocks remain; one subproblem per block
  // where each tile is wanted by itself
  const int run = tiles ? 1 : std::max(1, std::min(TC_RUN, p->pts.nsub / (3 * 4 * p->sms)));
  auto go = [&](auto k, size_t sm) {
    k<<<(p->pts.nsub + run - 1) / run, ST, sm, s>>>(
        (double*)p->fine, 2 * (z.n2 / 2 + 1), z.n1, z.n2, p->pts.nbins2, z.w, 1.0f / (float)((z.w + 2) / 2),
        p->pts.sub, p->pts.nsub, run, p->pts.cell, reinterpret_cast<const float2*>(p->pts.psi), p->pts.perm, d_map,
        tiles);
  };
  if (fine_products(p))
    go(spread_tc_k<true>, sizeof(SpreadSmem<ND + 1>));
  else
    go(spread_tc_k<false>, sizeof(SpreadSmem<ND>));
  NUSHT_CUDA(cudaGetLastError());
  return NUSHT_OK;
}

}  // namespace nusht
