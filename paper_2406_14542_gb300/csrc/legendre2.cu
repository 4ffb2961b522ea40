// legendre2.cu -- the iso-latitude step S and its adjoint in FP64 mode by the
// two-degree recurrence, the default of FP64 plans.
//
// Recurrence.  With x = cos(theta), eps_l^2 = (l^2 - m^2) / (4 l^2 - 1) and the
// orthonormal Pbar_l of order m, x Pbar_l = eps_{l+1} Pbar_{l+1} + eps_l Pbar_{l-1}.
// Applying it twice couples every other degree.  For the odd degrees
// l_i = m + 1 + 2 i the functions Pbar_{l_i} / x = s_i p_i (even polynomials in
// x times sin^m) obey, with scales s_i chosen so that the last coefficient is 1,
//   p_{i+1} = (a_i x^2 + b_i) p_i - p_{i-1},
//   s_{i+1} eps_{l+1} eps_{l+2} = s_{i-1} eps_l eps_{l-1}  (l = l_i),
//   a_i = s_i / (eps_{l+1} eps_{l+2} s_{i+1}),  b_i = -a_i (eps_{l+1}^2 + eps_l^2),
// and the even degrees are local combinations of them,
//   Pbar_{l_i - 1} = eps_{l_i} s_i p_i + eps_{l_i - 1} s_{i-1} p_{i-1}.
// So one chain of two FP64 multiply-adds serves two degrees, half of what the
// one-degree recurrence issues (this form is due to K. Ishioka, J. Meteorol.
// Soc. Japan 96, 2018).  Per order:
//   sum_{even} a_l Pbar_l = sum_i p_i E_i,  E_i = s_i (eps_{l_i} a_{l_i-1} + eps_{l_i+1} a_{l_i+1}),
//   sum_{odd}  a_l Pbar_l = x sum_i p_i O_i,  O_i = s_i a_{l_i}
// (E, O formed once per call, leg2_coef_k); the adjoint is the transpose:
// D_i = sum_rings p_i S_even and sum_rings p_i x S_odd, combined per degree by
// leg2_reduce_k.
//
// Accuracy.  In rings nearer the pole than theta = pi / 4 the step factor is
// formed as (a + b) - a sin^2(theta): sin^2 is exact to its last bit there
// while x^2 is not, and the phase error that x accumulates over thousands of
// degrees goes away.  Whole transforms at lmax 200 (kernel width 19) against sums
// in 128-bit floating point, one-degree -> this form: synthesis near the north
// pole off by at most 1.14e-13 -> 3.6e-14 of the largest value, over the sphere
// by 6.1e-14 -> 6.3e-14 of the norm, adjoint 6.1e-14 -> 6.3e-14, of a map in a
// polar cap 9.8e-14 -> 7.1e-14 (the FFT and NUFFT stages are most of it).
//
// Start of a chain.  A ring contributes to order m only from the degree where
// p_i first reaches 2^-74 (the sums flush smaller values; they are 2^-21 of a
// rounding error).  That step and the two values that continue the recurrence
// are found once at plan time (leg2_start_k, with scaled exponents), so a call
// neither forms sin^m(theta) nor runs the steps below: 0.69 of the full
// (ring pair, l, m) triples at lmax 4095 instead of the 0.86 that skipping
// whole 128-pair items leaves.
//
// Layout: one warp per (order, group of 32 ring pairs), in the adjoint per
// block of K groups, one pair per lane and group, two rings (theta, pi - theta)
// per pair through the parity of Pbar.  The sums run as float pairs on the FP32
// pipe (dfloat.cuh); per step and warp that is about 75 K issue slots under the
// 128 K cycles of the two DFMAs (one per 64 cycles), so the FP64 pipe is the bound.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <type_traits>
#include <vector>

#include "async_copy.cuh"
#include "ddouble.cuh"
#include "dfloat.cuh"
#include "nusht_internal.cuh"
#include "recurrence.cuh"

namespace nusht {

namespace {

using namespace rec;
constexpr unsigned FULL = 0xffffffffu;

struct Leg2Args {
  int lmax, mmax, M, npairs, ngrp, kblk;
  const double2* abx;  // (a_i, b_i): step factor a x^2 + b
  const double2* abs;  // (a_i, a_i + b_i): step factor a (-sin^2) + (a + b)
  const int* gst;      // [order][group of 32 pairs]: first step of any lane
  const int* ist;      // [order][pair]: first step of the pair (INT_MAX: never)
  const double2* st;   // [order][pair]: (p_i, p_{i-1}) at that step
  const double* ring_x;
  const double* ring_s;
};

// whether the rings of group g take the sin^2 form: uniform over the largest
// block of any kernel (32 kblk pairs), theta < pi / 4 at its middle
__device__ __forceinline__ bool polar(const Leg2Args& a, int g) {
  return (g / a.kblk) * a.kblk * 32 + a.kblk * 16 < a.npairs / 2;
}
__device__ __forceinline__ double step_arg(const Leg2Args& a, int j, bool pol) {
  const double v = pol ? __ldg(a.ring_s + j - 1) : __ldg(a.ring_x + j - 1);
  return pol ? -(v * v) : v * v;
}

// ---------------------------------------------------------------------------
// plan time: recurrence tables (double-double) and chain starts
// ---------------------------------------------------------------------------
// One warp per order.  The scales are a running product over every other step,
//   s_{i+1}^2 = s_{i-1}^2 (eps_l eps_{l-1})^2 / (eps_{l+1} eps_{l+2})^2,
// in double-double (numerators and denominators are exact integers below
// 2^53): each lane forms the factor of its step, a scan of stride two over the
// warp the products.
__global__ void __launch_bounds__(128) leg2_tab_k(int L, int mmax, double2* __restrict__ abx,
                                                  double2* __restrict__ abs, double* __restrict__ sc,
                                                  double* __restrict__ w1, double* __restrict__ w2) {
  const int lane = threadIdx.x & 31;
  const int m = blockIdx.x * 4 + (threadIdx.x >> 5);
  if (m > mmax) return;
  const int n = steps_of(L, m);
  const int64_t b0 = base_of(L, m);
  const double m2 = (double)m * m;
  auto num = [&](int l) { return (double)l * l - m2; };
  auto den = [&](int l) { return 4.0 * (double)l * l - 1.0; };
  // s_{i+1}^2 of the two steps before the chunk; s_0 = 1 / eps_{m+1} (p_0 = Pbar_mm), s_1 is free
  dd c0 = {1.0, 0.0}, c1 = dd_quot(den(m + 1), num(m + 1));
  for (int base = 0; base < n; base += 32) {
    const int i = base + lane, l = m + 1 + 2 * i;
    const double n0 = num(l), n1 = num(l + 1), n2 = num(l + 2), d0 = den(l), d1 = den(l + 1), d2 = den(l + 2);
    dd v;
    if (i == 0) {
      v = {c1.hi * sqrt((n0 / d0) / (n2 / d2)), 0.0};
    } else {
      v = dd_div(dd_div(dd_mul(dd_mul({n0, 0.0}, num(l - 1)), d1), n1), n2);
      v = dd_div(dd_div(dd_mul(v, d2), d0), den(l - 1));
    }
    for (int off = 2; off < 32; off *= 2) {
      const dd u = dd_up(v, off);
      if (lane >= off) v = dd_mul(v, u);
    }
    v = dd_mul(v, (lane & 1) ? c1 : c0);  // s_{i+1}^2
    dd s = dd_up(v, 1);                   // s_i^2
    if (lane == 0) s = c1;
    c0 = {__shfl_sync(FULL, v.hi, 30), __shfl_sync(FULL, v.lo, 30)};
    c1 = {__shfl_sync(FULL, v.hi, 31), __shfl_sync(FULL, v.lo, 31)};
    if (i >= n) continue;
    // a_i^2 = s_i^2 / (eps_{l+1}^2 eps_{l+2}^2 s_{i+1}^2)
    dd a2 = dd_div(dd_div(dd_mul(dd_mul(s, d1), d2), n1), n2);
    a2 = dd_div(a2, v.hi);  // the low word of the divisor to first order
    const double a = dd_root({a2.hi, a2.lo - a2.hi * (v.lo / v.hi)});
    const dd e = dd_add(dd_quot(n0, d0), dd_quot(n1, d1));  // eps_l^2 + eps_{l+1}^2
    const dd bx = dd_mul(e, -a), bs = dd_mul(dd_add({1.0, 0.0}, {-e.hi, -e.lo}), a);
    abx[b0 + i] = make_double2(a, bx.hi + bx.lo);
    abs[b0 + i] = make_double2(a, bs.hi + bs.lo);
    sc[b0 + i] = dd_root(s);
    w1[b0 + i] = dd_root(dd_div(dd_mul(s, n0), d0));  // s_i eps_{l_i}
    w2[b0 + i] = dd_root(dd_div(dd_mul(s, n1), d1));  // s_i eps_{l_i + 1}
  }
}

// One warp per (order, group of 32 pairs): each lane runs its chain from
// p_0 = c_m sin^m(theta) with a scaled exponent to the first step at or above
// 2^LEG2_TINY_EXP and keeps (p_i, p_{i-1}) there.
__global__ void __launch_bounds__(128) leg2_start_k(Leg2Args a, const double* __restrict__ cm, int* __restrict__ gst,
                                                    int* __restrict__ ist, double2* __restrict__ st) {
  const int lane = threadIdx.x & 31;
  const int it = blockIdx.x * 4 + (threadIdx.x >> 5);
  if (it >= (a.mmax + 1) * a.ngrp) return;
  const int m = it / a.ngrp, g = it % a.ngrp;
  const int j = g * 32 + lane + 1;
  const int n = steps_of(a.lmax, m);
  const bool pol = polar(a, g);
  const double2* tab = (pol ? a.abs : a.abx) + base_of(a.lmax, m);
  int first = INT_MAX;
  double q1 = 0.0, q2 = 0.0, z = 0.0;
  int E = 0;
  const bool valid = j <= a.npairs;
  if (valid) {
    z = step_arg(a, j, pol);
    double mant;
    int ex;
    pow_scaled(__ldg(a.ring_s + j - 1), m, mant, ex);
    const double q0 = __ldg(cm + m) * mant;
    E = ex >= LEG_TINY_EXP ? 0 : LEG_STEP_EXP * ((LEG_TINY_EXP - ex + LEG_STEP_EXP - 1) / LEG_STEP_EXP);
    q1 = q0 * exp2i(ex + E);
  }
  for (int i = 0; i < n; ++i) {
    if (valid && first == INT_MAX) {
      const int eb = (__double2hiint(q1) >> 20) & 0x7ff;
      if (E == 0 && eb >= 1023 + LEG2_TINY_EXP) {
        first = i;
      } else {
        const double2 ab = __ldg(tab + i);
        const double q = fma(fma(ab.x, z, ab.y), q1, -q2);
        q2 = q1;
        q1 = q;
        if (E != 0 && ((__double2hiint(q) >> 20) & 0x7ff) >= 1023 - 44) {
          q1 = scale_pow2(q1, -LEG_STEP_EXP);
          q2 = scale_pow2(q2, -LEG_STEP_EXP);
          E -= LEG_STEP_EXP;
        }
      }
    }
    if (__all_sync(FULL, !valid || first != INT_MAX)) break;
  }
  const size_t o = (size_t)m * a.ngrp * 32 + g * 32 + lane;
  ist[o] = first;
  st[o] = make_double2(q1, q2);
  const int mn = __reduce_min_sync(FULL, first);
  if (lane == 0) gst[it] = mn;
}

// ---------------------------------------------------------------------------
// per call: E_i, O_i from a_lm as float pairs, and the poles of order 0
// (Pbar_l0(0) = sqrt((2l+1)/4pi), Pbar_l0(pi) = (-1)^l of it) by the last
// row of blocks
// ---------------------------------------------------------------------------
__device__ __forceinline__ float4 pair4(double re, double im) {
  float4 r;
  df_of(re, r.x, r.y);
  df_of(im, r.z, r.w);
  return r;
}

__global__ void __launch_bounds__(256) leg2_coef_k(const double2* __restrict__ alm, int L, int mmax, int M,
                                                   const double* __restrict__ sc, const double* __restrict__ w1,
                                                   const double* __restrict__ w2,
                                                   const double* __restrict__ pole_norm, float4* __restrict__ eo,
                                                   double2* __restrict__ G) {
  const int m = blockIdx.y;
  if (m > mmax) {
    if (blockIdx.x) return;
    __shared__ double sn[256], ss[256];
    double nn = 0.0, sp = 0.0;
    for (int l = threadIdx.x; l <= L; l += 256) {
      const double v = alm[l].x * pole_norm[l];
      nn += v;
      sp += (l & 1) ? -v : v;
    }
    sn[threadIdx.x] = nn;
    ss[threadIdx.x] = sp;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
      if ((int)threadIdx.x < h) {
        sn[threadIdx.x] += sn[threadIdx.x + h];
        ss[threadIdx.x] += ss[threadIdx.x + h];
      }
      __syncthreads();
    }
    if (threadIdx.x == 0) {
      G[0] = make_double2(sn[0], 0.0);
      G[M / 2] = make_double2(ss[0], 0.0);
    }
    return;
  }
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= steps_of(L, m)) return;
  const int l = m + 1 + 2 * i;
  const double2* row = alm + mbase_of(L, m);
  const double2 z = make_double2(0.0, 0.0);
  double2 e0 = row[l - 1], o = l <= L ? row[l] : z, e1 = l + 1 <= L ? row[l + 1] : z;
  if (m == 0) e0.y = o.y = e1.y = 0.0;  // Im(a_l0) is ignored
  const int64_t k = base_of(L, m) + i;
  const double f0 = w1[k], f1 = w2[k], f = sc[k];
  eo[2 * k] = pair4(fma(f0, e0.x, f1 * e1.x), fma(f0, e0.y, f1 * e1.y));
  eo[2 * k + 1] = pair4(f * o.x, f * o.y);
}

// ---------------------------------------------------------------------------
// synthesis: one 32-pair group per warp; two or four pairs per lane share the
// coefficient reads but leave fewer warps and measured no faster at any size.
// At lmax 4095 19.9 ms, of which the two DFMAs per step take 18.9 ms of the
// FP64 pipe (the one-degree kernel: 52.0 ms).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(128) leg2_synth_k(Leg2Args a, const int* __restrict__ items, int nitems,
                                                    const float4* __restrict__ eo, double2* __restrict__ G) {
  const int lane = threadIdx.x & 31;
  const int it = blockIdx.x * 4 + (threadIdx.x >> 5);
  if (it >= nitems) return;
  const int v = __ldg(items + it);
  const int m = v >> 16, g = v & 0xffff;
  const int L = a.lmax, n = steps_of(L, m);
  const bool pol = polar(a, g);
  const int64_t b0 = base_of(L, m);
  const double2* tab = (pol ? a.abs : a.abx) + b0;
  const float4* ep = eo + 2 * b0;
  const size_t so = (size_t)m * a.ngrp * 32 + g * 32 + lane;
  const int jn = g * 32 + lane + 1;
  const double z = step_arg(a, min(jn, a.npairs), pol);
  const int is = __ldg(a.ist + so);
  const int i0 = __ldg(a.gst + m * a.ngrp + g);
  double q1 = 0.0, q2 = 0.0;
  float4 E = make_float4(0.f, 0.f, 0.f, 0.f), O = E;
  // the coefficients of 32 steps at a time through shared memory, the next 32
  // in flight: a warp that has the SM to itself would otherwise wait for an L2
  // read in every step (lmax 63: 10.8 -> 7.9 us; lmax 4095: 21.3 -> 19.9 ms)
  __shared__ double2 s_ab[4][2][32];
  __shared__ float4 s_eo[4][2][64];
  double2(*ba)[32] = s_ab[threadIdx.x >> 5];
  float4(*be)[64] = s_eo[threadIdx.x >> 5];
  auto fetch = [&](int c, int buf) {
    copy16(&ba[buf][lane], tab + min(c + lane, n - 1));
    copy16(&be[buf][lane], ep + min(2 * c + lane, 2 * n - 1));
    copy16(&be[buf][lane + 32], ep + min(2 * c + lane + 32, 2 * n - 1));
  };
  fetch(i0, 0);
  copies_commit();
  int buf = 0;
  for (int c = i0; c < n; c += 32, buf ^= 1) {
    if (c + 32 < n) fetch(c + 32, buf ^ 1);
    copies_commit();
    copies_wait<1>();
    __syncwarp();
    const int ns = min(32, n - c);
    for (int t = 0; t < ns; ++t) {
      const double2 ab = ba[buf][t];
      const float4 ce = be[buf][2 * t], co = be[buf][2 * t + 1];
      if (c + t == is) {
        const double2 s = __ldg(a.st + so);
        q1 = s.x;
        q2 = s.y;
      }
      const double q = fma(fma(ab.x, z, ab.y), q1, -q2);
      float qh, ql;
      split_qr(q1, qh, ql);
      q2 = q1;
      q1 = q;
      df_mac(E.x, E.y, ce.x, ce.y, qh, ql);
      df_mac(E.z, E.w, ce.z, ce.w, qh, ql);
      df_mac(O.x, O.y, co.x, co.y, qh, ql);
      df_mac(O.z, O.w, co.z, co.w, qh, ql);
    }
    __syncwarp();  // the buffer is refilled by the next chunk
  }
  if (jn > a.npairs) return;
  // F(theta_j) = E + x O, F(pi - theta_j) = E - x O, doubled with (-1)^m
  const int M = a.M, js = M / 2 - jn;
  const double sg = (m & 1) ? -1.0 : 1.0;
  double2* row = G + (size_t)m * M;
  const double x = __ldg(a.ring_x + jn - 1);
  const double er = df_value(E.x, E.y), ei = df_value(E.z, E.w);
  const double orr = x * df_value(O.x, O.y), oi = x * df_value(O.z, O.w);
  const double2 fn = make_double2(er + orr, ei + oi);
  const double2 fs = make_double2(er - orr, ei - oi);
  row[jn] = fn;
  row[M - jn] = make_double2(sg * fn.x, sg * fn.y);
  if (js != jn) {
    row[js] = fs;
    row[M - js] = make_double2(sg * fs.x, sg * fs.y);
  }
}

// ---------------------------------------------------------------------------
// adjoint: partial[block][2 k, 2 k + 1] = sum over the block's rings of
// p_i (S_even, x S_odd).  Each step's sums over the lane's K chains go to two
// shared-memory slots; every four steps the warp sums the slots over its 32
// lanes through the transpose: lane t sums one float pair (slot t / 4, re or
// im) over 16 lanes, one shuffle joins the halves.  K spreads that reduction
// over more pairs but makes fewer warps (see leg2_setup).  A lane's sums have
// at most four terms, so they stay open (dfloat.cuh) until the transpose
// renormalises them: 21.4 against 23.0 ms at lmax 4095, where the FP64 pipe's
// share is 18.9 ms (the one-degree kernel: 52.6 ms).
// ---------------------------------------------------------------------------
template <int K>
__global__ void __launch_bounds__(128, 6) leg2_adj_k(Leg2Args a, const int* __restrict__ items, int nitems,
                                                  const double2* __restrict__ Gt, float4* __restrict__ partial,
                                                  int64_t n2) {
  // folded spectrum of the lane's chains, even and x odd, as float pairs; the
  // slots of a lane are padded to nine (conflict-free 16-byte stores)
  __shared__ float4 sS[2][K][128];
  __shared__ float4 red[4][32][9];
  // step coefficients as in the synthesis; with four pairs per lane one step
  // lasts 512 cycles and a read one step ahead is enough (22.9 against 23.4 ms
  // at lmax 4095; with two pairs 566 against 546 us at lmax 1023)
  constexpr bool STAGED = K < 4;
  __shared__ double2 s_ab[STAGED ? 4 : 1][2][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int it = blockIdx.x * 4 + warp;
  if (it >= nitems) return;
  const int v = __ldg(items + it);
  const int m = v >> 16, blk = v & 0xffff, g0 = blk * K;
  const int L = a.lmax, n = steps_of(L, m), M = a.M;
  const bool pol = polar(a, g0);
  const int64_t b0 = base_of(L, m);
  const double2* tab = (pol ? a.abs : a.abx) + b0;
  const size_t so = (size_t)m * a.ngrp * 32 + g0 * 32 + lane;
  const double sg = (m & 1) ? -1.0 : 1.0;
  const double2* row = Gt + (size_t)m * M;
  float4(*rw)[9] = red[warp];
  float4* SE = &sS[0][0][threadIdx.x];
  float4* SO = &sS[1][0][threadIdx.x];
  int gs[K], is[K];
  double q1[K], q2[K], z[K];
  int i0 = INT_MAX;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const bool have = g0 + k < a.ngrp;
    gs[k] = have ? __ldg(a.gst + m * a.ngrp + g0 + k) : INT_MAX;
    is[k] = have ? __ldg(a.ist + so + k * 32) : INT_MAX;
    const int jn = (g0 + k) * 32 + lane + 1;
    z[k] = step_arg(a, min(jn, a.npairs), pol);
    q1[k] = q2[k] = 0.0;
    i0 = min(i0, gs[k]);
    // D^dagger: F(theta_j) = G(theta_j) + (-1)^m G(2 pi - theta_j)
    double2 fn = make_double2(0.0, 0.0), fs = fn;
    double x = 0.0;
    if (gs[k] != INT_MAX && jn <= a.npairs) {
      const int js = M / 2 - jn;
      x = __ldg(a.ring_x + jn - 1);
      const double2 u0 = row[jn], u1 = row[M - jn];
      fn = make_double2(u0.x + sg * u1.x, u0.y + sg * u1.y);
      if (js != jn) {
        const double2 h0 = row[js], h1 = row[M - js];
        fs = make_double2(h0.x + sg * h1.x, h0.y + sg * h1.y);
      }
    }
    SE[k * 128] = pair4(fn.x + fs.x, fn.y + fs.y);
    SO[k * 128] = pair4(x * (fn.x - fs.x), x * (fn.y - fs.y));
  }
  if (i0 >= n) return;
  float4* out = partial + (size_t)blk * 2 * n2 + 2 * b0;
  const int d = lane >> 2, cpt = (lane >> 1) & 1, half = lane & 1;
  double2(*ba)[32] = s_ab[STAGED ? warp : 0];
  auto fetch = [&](int c, int buf) {
    copy16(&ba[buf][lane], tab + min(c + lane, n - 1));
    copies_commit();
  };
  double2 ab = make_double2(0.0, 0.0);
  if (STAGED)
    fetch(i0, 0);
  else
    ab = __ldg(tab + i0);
  for (int base = i0; base < n; base += 4) {
    const int at = base - i0, buf = (at >> 5) & 1;
    if (STAGED && (at & 31) == 0) {
      fetch(base + 32, buf ^ 1);
      copies_wait<1>();
      __syncwarp();
    }
    const int ns = min(4, n - base);
#pragma unroll 1
    for (int t = 0; t < ns; ++t) {
      const int i = base + t;
      double2 abn = ab;
      if (STAGED)
        ab = ba[buf][(at & 31) + t];
      else
        abn = __ldg(tab + min(i + 1, n - 1));
      float4 e, o;
      // the group nearest the equator starts first: it opens the step's sums
#pragma unroll
      for (int k = K - 1; k >= 0; --k) {
        if (k < K - 1 && i < gs[k]) continue;  // warp-uniform
        if (i == is[k]) {
          const double2 s = __ldg(a.st + so + k * 32);
          q1[k] = s.x;
          q2[k] = s.y;
        }
        const double q = fma(fma(ab.x, z[k], ab.y), q1[k], -q2[k]);
        float qh, ql;
        split_qr(q1[k], qh, ql);
        q2[k] = q1[k];
        q1[k] = q;
        const float4 se = SE[k * 128], sd = SO[k * 128];
        if (k == K - 1) {
          df_prod(e.x, e.y, se.x, se.y, qh, ql);
          df_prod(e.z, e.w, se.z, se.w, qh, ql);
          df_prod(o.x, o.y, sd.x, sd.y, qh, ql);
          df_prod(o.z, o.w, sd.z, sd.w, qh, ql);
        } else {
          df_mac_open(e.x, e.y, se.x, se.y, qh, ql);
          df_mac_open(e.z, e.w, se.z, se.w, qh, ql);
          df_mac_open(o.x, o.y, sd.x, sd.y, qh, ql);
          df_mac_open(o.z, o.w, sd.z, sd.w, qh, ql);
        }
      }
      if (!STAGED) ab = abn;
      rw[lane][2 * t] = e;
      rw[lane][2 * t + 1] = o;
    }
    __syncwarp();
    float sh = 0.f, sl = 0.f;
    if (d < 2 * ns) {
#pragma unroll 4
      for (int i = 0; i < 16; ++i) {
        const float2 x = reinterpret_cast<const float2*>(&rw[half * 16 + i][d])[cpt];
        df_add(sh, sl, x.x, x.y);
      }
    }
    const float oh = __shfl_xor_sync(FULL, sh, 1), ol = __shfl_xor_sync(FULL, sl, 1);
    df_add(sh, sl, oh, ol);
    __syncwarp();  // the slots are rewritten by the next four steps
    if (half == 0 && d < 2 * ns) reinterpret_cast<float2*>(out + 2 * base + d)[cpt] = make_float2(sh, sl);
  }
  if (STAGED) copies_wait<0>();  // the chunk past the last one
}

// c_lm from the block partials (summed as float pairs in a fixed order, only
// the blocks that have started at step i): odd degrees s_i D^O_i, even degrees
// w1_i D^E_i + w2_{i-1} D^E_{i-1}; the poles join order 0.  wpos multiplies
// the m > 0 entries (1: the adjoint, 2: the gradient of a real loss).
__global__ void __launch_bounds__(256) leg2_reduce_k(Leg2Args a, int K, int nblk, const float4* __restrict__ partial,
                                                     int64_t n2, const double* __restrict__ sc,
                                                     const double* __restrict__ w1, const double* __restrict__ w2,
                                                     const double* __restrict__ pole_norm,
                                                     const double2* __restrict__ Gt, double wpos,
                                                     double2* __restrict__ out) {
  __shared__ double2 ev[257];
  __shared__ int start[256];  // first step of each block (at most 256: lmax <= 16383)
  const int m = blockIdx.y, L = a.lmax, n = steps_of(L, m);
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (blockIdx.x * 256 >= n) return;
  const int64_t b0 = base_of(L, m);
  if ((int)threadIdx.x < nblk) {
    int g = INT_MAX;
    for (int k = threadIdx.x * K; k < min((int)(threadIdx.x + 1) * K, a.ngrp); ++k)
      g = min(g, __ldg(a.gst + m * a.ngrp + k));
    start[threadIdx.x] = g;
  }
  __syncthreads();
  auto sums = [&](int s, double2* even, double2* odd) {
    float4 e = make_float4(0.f, 0.f, 0.f, 0.f), o = e;
    for (int b = 0; b < nblk; ++b) {
      if (s < start[b]) continue;
      const float4* p = partial + (size_t)b * 2 * n2 + 2 * (b0 + s);
      const float4 x = p[0];
      df_add(e.x, e.y, x.x, x.y);
      df_add(e.z, e.w, x.z, x.w);
      if (odd) {
        const float4 y = p[1];
        df_add(o.x, o.y, y.x, y.y);
        df_add(o.z, o.w, y.z, y.w);
      }
    }
    *even = make_double2(df_value(e.x, e.y), df_value(e.z, e.w));
    if (odd) *odd = make_double2(df_value(o.x, o.y), df_value(o.z, o.w));
  };
  double2 de = make_double2(0.0, 0.0), od = de;
  if (i < n) sums(i, &de, &od);
  ev[threadIdx.x + 1] = de;
  if (threadIdx.x == 0) {
    double2 h = make_double2(0.0, 0.0);
    if (i > 0) sums(i - 1, &h, nullptr);
    ev[0] = h;
  }
  __syncthreads();
  if (i >= n) return;
  const int64_t k = b0 + i;
  const double2 dp = ev[threadIdx.x];
  const double f0 = w1[k], f1 = i > 0 ? w2[k - 1] : 0.0, f = sc[k];
  double2 ce = make_double2(fma(f0, de.x, f1 * dp.x), fma(f0, de.y, f1 * dp.y));
  double2 co = make_double2(f * od.x, f * od.y);
  const int l = m + 2 * i;
  double2* row = out + mbase_of(L, m);
  if (m == 0) {  // real
    const double np = Gt[0].x, sp = Gt[a.M / 2].x;
    ce = make_double2(ce.x + pole_norm[l] * (np + sp), 0.0);
    if (l + 1 <= L) co = make_double2(co.x + pole_norm[l + 1] * (np - sp), 0.0);
  } else {
    ce = make_double2(wpos * ce.x, wpos * ce.y);
    co = make_double2(wpos * co.x, wpos * co.y);
  }
  row[l] = ce;
  if (l + 1 <= L) row[l + 1] = co;
}

Leg2Args args_of(nusht_plan_t p) {
  Leg2Args a;
  a.lmax = p->lmax;
  a.mmax = p->mmax;
  a.M = p->sz.M;
  a.npairs = p->leg.npairs;
  a.ngrp = (a.npairs + 31) / 32;
  a.kblk = p->leg2.ka;
  a.abx = p->leg2.abx;
  a.abs = p->leg2.abs;
  a.gst = p->leg2.gst;
  a.ist = p->leg2.ist;
  a.st = p->leg2.st;
  a.ring_x = p->leg.ring_x;
  a.ring_s = p->leg.ring_s;
  return a;
}

}  // namespace

int64_t leg2_entries(int lmax, int mmax) { return base_of(lmax, mmax + 1); }

// Needs the ring tables, cm and pole_norm of legendre_build_tables.
int leg2_setup(nusht_plan_t p, cudaStream_t s) {
  Leg2Tables& t = p->leg2;
  const int L = p->lmax, mmax = p->mmax;
  t.n2 = leg2_entries(L, mmax);
  const int ngrp = (p->leg.npairs + 31) / 32;
  // the adjoint's pairs per lane, by the number of (order, group) chains; with
  // 1 / 2 / 4, kernel and partial reduction take 104 / 131 / 240 us at 2,700
  // (lmax 517, mmax 301), 471 / 463 / 624 at 16,400 (lmax 1023), 3,200 / 2,950 /
  // 3,030 at 65,500 (lmax 2047), 23.8 / 21.7 / 21.7 ms at 262,000 (lmax 4095),
  // where four also halve the partial rows (2.2 GB)
  const int64_t groups = (int64_t)(mmax + 1) * ngrp;
  t.ka = groups < LEG2_GROUPS_K1 ? 1 : groups < LEG2_GROUPS_K2 ? 2 : 4;
  const size_t n2 = (size_t)t.n2, np = (size_t)(mmax + 1) * ngrp * 32;
  // one allocation: at small lmax a plan costs what its allocations cost
  char* at = nullptr;
  auto carve = [&](auto*& q, size_t n) {
    q = reinterpret_cast<std::remove_reference_t<decltype(q)>>(at);
    at += (n * sizeof(*q) + 255) / 256 * 256;
  };
  auto layout = [&]() {
    carve(t.abx, n2);
    carve(t.abs, n2);
    carve(t.st, np);
    carve(t.sc, n2);
    carve(t.w1, n2);
    carve(t.w2, n2);
    carve(t.ist, np);
    carve(t.gst, (size_t)groups);
    carve(t.items_s, (size_t)groups);
    carve(t.items_a, (size_t)groups);
  };
  layout();
  NUSHT_TRY(dev_alloc(&t.slab, (size_t)at, &p->bytes));
  at = (char*)t.slab;
  layout();
  leg2_tab_k<<<(mmax + 4) / 4, 128, 0, s>>>(L, mmax, t.abx, t.abs, t.sc, t.w1, t.w2);
  leg2_start_k<<<(int)((groups + 3) / 4), 128, 0, s>>>(args_of(p), p->leg.cm, t.gst, t.ist, t.st);
  NUSHT_CUDA(cudaGetLastError());
  std::vector<int> gst((size_t)groups);
  NUSHT_CUDA(cudaMemcpyAsync(gst.data(), t.gst, gst.size() * 4, cudaMemcpyDeviceToHost, s));
  NUSHT_CUDA(cudaStreamSynchronize(s));
  // work lists, one entry (order << 16 | block) per block with a started ring;
  // orders ascend, so the longest chains are issued first
  auto list = [&](int K, std::vector<int>& v) {
    for (int m = 0; m <= mmax; ++m)
      for (int b = 0; b * K < ngrp; ++b) {
        int g = INT_MAX;
        for (int k = b * K; k < std::min((b + 1) * K, ngrp); ++k) g = std::min(g, gst[(size_t)m * ngrp + k]);
        if (g != INT_MAX) v.push_back((m << 16) | b);
      }
  };
  std::vector<int> is, ia;
  list(1, is);
  list(t.ka, ia);
  t.nis = (int)is.size();
  t.nia = (int)ia.size();
  NUSHT_CUDA(cudaMemcpyAsync(t.items_s, is.data(), is.size() * 4, cudaMemcpyHostToDevice, s));
  NUSHT_CUDA(cudaMemcpyAsync(t.items_a, ia.data(), ia.size() * 4, cudaMemcpyHostToDevice, s));
  NUSHT_CUDA(cudaStreamSynchronize(s));
  p->leg.nitems = t.nis;
  p->leg.nitems_total = (mmax + 1) * ngrp;
  int64_t tri = 0;
  for (int m = 0; m <= mmax; ++m)
    for (int g = 0; g < ngrp; ++g)
      if (const int f = gst[(size_t)m * ngrp + g]; f != INT_MAX)
        tri += (int64_t)std::min(32, p->leg.npairs - g * 32) * (L - m + 1 - 2 * f);
  p->leg.triples = tri;
  return NUSHT_OK;
}

size_t leg2_partial_bytes(nusht_plan_t p) {
  const int ngrp = (p->leg.npairs + 31) / 32;
  return (size_t)((ngrp + p->leg2.ka - 1) / p->leg2.ka) * 2 * (size_t)p->leg2.n2 * sizeof(float4);
}

void leg2_free(nusht_plan_t p) {
  Leg2Tables& t = p->leg2;
  dev_free(t.slab);
  t = Leg2Tables();
}

int leg2_synth(nusht_plan_t p, const void* d_alm, cudaStream_t s) {
  const Leg2Tables& t = p->leg2;
  const Leg2Args a = args_of(p);
  float4* eo = (float4*)p->atilde;
  double2* G = (double2*)p->G;
  const dim3 cg((steps_of(p->lmax, 0) + 255) / 256, p->mmax + 2);
  leg2_coef_k<<<cg, 256, 0, s>>>((const double2*)d_alm, p->lmax, p->mmax, a.M, t.sc, t.w1, t.w2, p->leg.pole_norm, eo,
                                 G);
  if (t.nis > 0) leg2_synth_k<<<(t.nis + 3) / 4, 128, 0, s>>>(a, t.items_s, t.nis, eo, G);
  NUSHT_CUDA(cudaGetLastError());
  return NUSHT_OK;
}

int leg2_adjoint(nusht_plan_t p, void* d_alm, cudaStream_t s, double wpos) {
  const Leg2Tables& t = p->leg2;
  const Leg2Args a = args_of(p);
  const double2* Gt = (const double2*)p->Ghat;
  float4* part = (float4*)p->partial;
  const int nb = (t.nia + 3) / 4;
  if (nb > 0) {
    if (t.ka == 1)
      leg2_adj_k<1><<<nb, 128, 0, s>>>(a, t.items_a, t.nia, Gt, part, t.n2);
    else if (t.ka == 2)
      leg2_adj_k<2><<<nb, 128, 0, s>>>(a, t.items_a, t.nia, Gt, part, t.n2);
    else
      leg2_adj_k<4><<<nb, 128, 0, s>>>(a, t.items_a, t.nia, Gt, part, t.n2);
  }
  const dim3 rg((steps_of(p->lmax, 0) + 255) / 256, p->mmax + 1);
  leg2_reduce_k<<<rg, 256, 0, s>>>(a, t.ka, (a.ngrp + t.ka - 1) / t.ka, part, t.n2, t.sc, t.w1, t.w2,
                                   p->leg.pole_norm, Gt, wpos, (double2*)d_alm);
  NUSHT_CUDA(cudaGetLastError());
  return NUSHT_OK;
}

}  // namespace nusht
