// spin.cu -- spin-weighted transforms (the spin-n generalisation named in the
// Conclusion, Sec. 5) through the same double Fourier sphere chain.
//
// For spin s >= 1 two real fields Q, U carry Q + i U = sum (G_lm + i C_lm) sY_lm
// with sY_lm = (-1)^s sqrt((2l+1)/(4 pi)) d^l_{m,-s}(theta) e^{i m phi} and G, C
// real-field coefficients (stored for m >= 0).  With
//   lambda+ = sY_lm(theta, 0),  lambda- = (-s)Y_lm(theta, 0),
//   W = (lambda+ + (-1)^s lambda-) / 2,  X = (lambda+ - (-1)^s lambda-) / 2,
// the iso-latitude step gives for each order the two ring functions
//   F^Q_m = sum_l (G_lm W + i C_lm X),   F^U_m = sum_l (C_lm W - i G_lm X),
// and Q, U are real-field syntheses of F^Q, F^U (F_0 + 2 Re sum_{m>0} F_m e^{imphi}).
// The doubling D carries one more sign: a spin-s quantity changes sign
// (-1)^s with the local frame on the continuation through the pole, so
// G(2 pi - theta) = (-1)^(m+s) F(theta).
//
// Legendre part.  For each (order m, ring pair theta, pi - theta) two Wigner-d
// recurrences in l run in FP64 (pv = lambda+ ~ d^l_{m,-s}, nv = lambda- ~
// d^l_{m,s}).  With beta_l^2 = (l^2 - m^2) (l^2 - s^2) / (l^2 (4 l^2 - 1)),
//   x v_l = beta_{l+1} v_{l+1} -/+ m s / (l (l+1)) v_l + beta_l v_{l-1};
// writing v_l = s_l p_l with s_{l+1} beta_{l+1} = s_{l-1} beta_l makes the last
// coefficient 1,
//   p_{l+1} = (a_l x +/- b_l) p_l - p_{l-1},  a_l = s_l / (beta_{l+1} s_{l+1}),  b_l = a_l m s / (l (l+1)),
// two FP64 multiply-adds per chain and degree (the unscaled form needs three
// operations).  Nearer the pole than pi / 4 the factor is formed as
// (a +/- b) - 2 a sin^2(theta / 2), which keeps the last bits that x loses
// there.  The scales go into the coefficients (synthesis) and into the sums
// over the rings (adjoint).  Since d^l_{m,-s}(pi - theta) = (-1)^(l+m)
// d^l_{m,s}(theta), the two chains at theta give both rings: with
// p = (-1)^(l+m+s), pv(pi - theta) = p (-1)^s nv and nv(pi - theta) =
// p (-1)^s pv.  In terms of A+ = (G + iC) / 2 and A- = (-1)^s (G - iC) / 2,
//   north: F^Q = sum pv A+ + nv A-,   F^U = -i (sum pv A+ - nv A-),
//   south: F^Q = (-1)^s sum p (nv A+ + pv A-),  F^U = (-1)^s i sum p (pv A- - nv A+),
// four complex sums per ring pair, kept as float pairs on the FP32 pipe
// (the FP64 pipe carries only the four recurrence operations per degree).
// The adjoint is the transpose: with B+- = H^Q +- i H^U at each ring,
// U1 = (B+_n + p B-_s) / 2, U2 = (-1)^s (B-_n + p B+_s) / 2 and V1, V2 with
// -p, each degree adds G = pv U1 + nv U2 and C = i (nv V2 - pv V1) per ring
// pair; the lanes' float-pair sums go to shared-memory slots and every four
// degrees the warp reduces them through a transpose (lane t sums one float
// pair over 16 lanes, one shuffle joins the halves).
//
// Work and starts.  One warp per (order, group of 32 ring pairs), one pair per
// lane, one partial row per group in the adjoint, summed in a fixed order.  As
// in legendre2.cu the degree where each chain first reaches 2^-74 and the two
// values that continue it are found once at plan time (with scaled
// exponents); a call starts there, and a group where nothing starts
// costs nothing (synthesis writes its rings as zeros).
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
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

struct SpinArgs {
  int lmax, mmax, M, npairs, ngrp, s;
  const double2* ab[2];  // per packed (l, m): (a, b) for x, (a, a + b) for -2 sin^2(theta / 2)
  const double* bm[2];   // the same for the lambda- chain: -b, a - b
  const int* gst;        // [order][group]: first degree of any chain
  const int* ist;        // [chain][order][pair]: first degree (INT_MAX: never)
  const double2* st;     // [chain][order][pair]: (p_l, p_{l-1}) there
};

__device__ __forceinline__ bool spin_polar(const SpinArgs& a, int g) { return g * 32 + 16 < a.npairs / 2; }
// argument of the step factor: x, or x - 1 = -2 sin^2(theta / 2); theta = 2 pi j / M
__device__ __forceinline__ double spin_arg(const SpinArgs& a, int j, bool pol) {
  if (!pol) return cospi(2.0 * (double)j / (double)a.M);
  const double h = sinpi((double)j / (double)a.M);
  return -2.0 * h * h;
}

// plan time: one warp per (order, group): each lane runs its two chains to
// their first value at or above 2^LEG2_TINY_EXP
__global__ void __launch_bounds__(128) spin_start_k(SpinArgs a, const double* __restrict__ st_mant,
                                                    const int* __restrict__ st_exp, const int* __restrict__ st_ab,
                                                    int* __restrict__ gst, int* __restrict__ ist,
                                                    double2* __restrict__ st) {
  const int lane = threadIdx.x & 31;
  const int it = blockIdx.x * 4 + (threadIdx.x >> 5);
  if (it >= (a.mmax + 1) * a.ngrp) return;
  const int m = it / a.ngrp, g = it % a.ngrp;
  const int j = g * 32 + lane + 1, L = a.lmax;
  const int l0 = m > a.s ? m : a.s;
  const bool pol = spin_polar(a, g), valid = j <= a.npairs;
  const int mb = mbase_of(L, m);
  const size_t np = (size_t)(a.mmax + 1) * a.ngrp * 32, o = (size_t)m * a.ngrp * 32 + g * 32 + lane;
  const double z = spin_arg(a, min(j, a.npairs), pol);
  double sh, chh;
  sincospi((double)min(j, a.npairs) / (double)a.M, &sh, &chh);  // theta / 2 = pi j / M
  int mn = INT_MAX;
  for (int c = 0; c < 2; ++c) {
    int first = INT_MAX, E = 0;
    double q1 = 0.0, q2 = 0.0;
    if (valid && l0 <= L) {
      const int pw = __ldg(st_ab + 2 * m + c);
      double ma, mb2;
      int ea, eb;
      pow_scaled(chh, pw >> 16, ma, ea);
      pow_scaled(sh, pw & 0xffff, mb2, eb);
      const double v = __ldg(st_mant + 2 * m + c) * ma * mb2;  // mantissas in [0.25, 1) x [0.5, 1)
      const int e = __ldg(st_exp + 2 * m + c) + ea + eb;
      E = e >= LEG_TINY_EXP ? 0 : LEG_STEP_EXP * ((LEG_TINY_EXP - e + LEG_STEP_EXP - 1) / LEG_STEP_EXP);
      q1 = v * exp2i(e + E);
    }
    for (int l = l0; l <= L; ++l) {
      if (valid && first == INT_MAX) {
        const int eb = (__double2hiint(q1) >> 20) & 0x7ff;
        if (E == 0 && eb >= 1023 + LEG2_TINY_EXP) {
          first = l;
        } else {
          const double2 ab = __ldg((pol ? a.ab[1] : a.ab[0]) + mb + l);
          const double f = fma(ab.x, z, c ? __ldg((pol ? a.bm[1] : a.bm[0]) + mb + l) : ab.y);
          const double q = fma(f, q1, -q2);
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
    ist[c * np + o] = first;
    st[c * np + o] = make_double2(q1, q2);
    mn = min(mn, (int)__reduce_min_sync(FULL, first));
  }
  if (lane == 0) gst[it] = mn;
}

// plan time: step coefficients and scales, one warp per order; the scales are
// a running product over every other degree (s_{l+1}^2 = s_{l-1}^2 beta_l^2 /
// beta_{l+1}^2) in double-double, scanned over the warp as in legendre2.cu
__global__ void __launch_bounds__(128) spin_tab_k(int L, int mmax, int sp, double2* __restrict__ abx,
                                                  double* __restrict__ bmx, double2* __restrict__ abs,
                                                  double* __restrict__ bms, double* __restrict__ sc) {
  const int lane = threadIdx.x & 31;
  const int m = blockIdx.x * 4 + (threadIdx.x >> 5);
  if (m > mmax) return;
  const int l0 = m > sp ? m : sp;
  if (l0 > L) return;
  const int mb = mbase_of(L, m);
  const double m2 = (double)m * m, s2 = (double)sp * sp;
  // v beta_l^2 and v / beta_l^2 factor by factor (every factor is exact)
  auto mulb = [&](dd v, int l) {
    const double q = (double)l * l;
    return dd_div(dd_div(dd_mul(dd_mul(v, q - m2), q - s2), q), 4.0 * q - 1.0);
  };
  auto divb = [&](dd v, int l) {
    const double q = (double)l * l;
    return dd_div(dd_div(dd_mul(dd_mul(v, q), 4.0 * q - 1.0), q - m2), q - s2);
  };
  dd c0 = {1.0, 0.0}, c1 = {1.0, 0.0};  // lanes 30, 31 of the chunk before; s_{l0} = 1
  for (int base = l0; base <= L; base += 32) {
    const int l = base + lane;
    dd v;  // factor of s_{l+1}^2
    if (l == l0) {
      // s_{l0+1} is free: (beta_{l0+1} / beta_{l0+2})^(1/2) evens out the steps
      v = {sqrt(divb(mulb({1.0, 0.0}, l0 + 1), l0 + 2).hi), 0.0};
    } else {
      v = divb(mulb({1.0, 0.0}, l), l + 1);
    }
    for (int off = 2; off < 32; off *= 2) {
      const dd u = dd_up(v, off);
      if (lane >= off) v = dd_mul(v, u);
    }
    v = dd_mul(v, (lane & 1) ? c1 : c0);  // s_{l+1}^2
    dd s = dd_up(v, 1);                   // s_l^2
    if (lane == 0) s = c1;
    c0 = {__shfl_sync(FULL, v.hi, 30), __shfl_sync(FULL, v.lo, 30)};
    c1 = {__shfl_sync(FULL, v.hi, 31), __shfl_sync(FULL, v.lo, 31)};
    if (l > L) continue;
    dd a2 = divb(s, l + 1);
    a2 = dd_div(a2, v.hi);  // the low word of the divisor to first order
    const double a = dd_root({a2.hi, a2.lo - a2.hi * (v.lo / v.hi)});
    const dd r = dd_quot((double)m * sp, (double)l * (l + 1.0));
    const dd b = dd_mul(r, a);
    const dd p = dd_mul(dd_add({1.0, 0.0}, r), a), n = dd_mul(dd_add({1.0, 0.0}, {-r.hi, -r.lo}), a);
    abx[mb + l] = make_double2(a, b.hi + b.lo);
    bmx[mb + l] = -(b.hi + b.lo);
    abs[mb + l] = make_double2(a, p.hi + p.lo);
    bms[mb + l] = n.hi + n.lo;
    sc[mb + l] = dd_root(s);
  }
}

// s_l (G + iC) / 2 and s_l (-1)^s (G - iC) / 2 per packed (l, m) as float pairs
// (hi re, lo re, hi im, lo im); Im of the m = 0 entries is ignored
__global__ void spin_scale_k(const double2* __restrict__ glm, const double2* __restrict__ clm,
                             const double* __restrict__ sc, int64_t nalm, int L, int s, float4* __restrict__ ap,
                             float4* __restrict__ am) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nalm) return;
  double2 g = glm[i], c = clm[i];
  if (i <= L) g.y = c.y = 0.0;
  const double f = 0.5 * sc[i], hs = (s & 1) ? -f : f;  // entries below degree s: scale 0
  float4 p, q;
  df_of(f * (g.x - c.y), p.x, p.y);
  df_of(f * (g.y + c.x), p.z, p.w);
  df_of(hs * (g.x + c.y), q.x, q.y);
  df_of(hs * (g.y - c.x), q.z, q.w);
  ap[i] = p;
  am[i] = q;
}

// acc += (float-pair complex a) * (float-pair real v)
__device__ __forceinline__ void cmac(float4& acc, const float4 a, float vh, float vl) {
  df_mac(acc.x, acc.y, a.x, a.y, vh, vl);
  df_mac(acc.z, acc.w, a.z, a.w, vh, vl);
}

// the first product of a sum, and the next (dfloat.cuh: open sums)
__device__ __forceinline__ void cprod(float4& acc, const float4 a, float vh, float vl) {
  df_prod(acc.x, acc.y, a.x, a.y, vh, vl);
  df_prod(acc.z, acc.w, a.z, a.w, vh, vl);
}
__device__ __forceinline__ void cmac_open(float4& acc, const float4 a, float vh, float vl) {
  df_mac_open(acc.x, acc.y, a.x, a.y, vh, vl);
  df_mac_open(acc.z, acc.w, a.z, a.w, vh, vl);
}

__device__ __forceinline__ double2 cval(const float4 v) {
  return make_double2(df_value(v.x, v.y), df_value(v.z, v.w));
}

// A warp's 32-degree chunks of step coefficients (synthesis: and of A+, A-) in
// shared memory, the next chunk in flight.  Degrees run in pairs of parity
// l + m + s even, odd, so a chunk may begin one degree below the first
// (clamped: nothing has started there).
struct SpinChunk {
  double2 ab[32];
  double bm[32];
};

// synthesis: the Q and U ring maps, doubled, [m][M] complex each
__global__ void __launch_bounds__(128) spin_synth_k(SpinArgs a, const float4* __restrict__ ap,
                                                    const float4* __restrict__ am, double2* __restrict__ GQ,
                                                    double2* __restrict__ GU) {
  __shared__ __align__(16) SpinChunk s_t[4][2];
  __shared__ float4 s_c[4][2][64];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int it = blockIdx.x * 4 + warp;
  if (it >= (a.mmax + 1) * a.ngrp) return;
  const int m = it / a.ngrp, g = it % a.ngrp;
  const int L = a.lmax, s = a.s, M = a.M;
  const int l0 = m > s ? m : s;
  const int jn = g * 32 + lane + 1, js = M / 2 - jn;
  double2* rq = GQ + (size_t)m * M;
  double2* ru = GU + (size_t)m * M;
  const int ls = __ldg(a.gst + it);
  if (ls > L) {  // nothing starts: the rings are zero (the adjoint writes these buffers)
    if (jn <= a.npairs) {
      const double2 o = make_double2(0.0, 0.0);
      rq[jn] = ru[jn] = rq[M - jn] = ru[M - jn] = o;
      rq[js] = ru[js] = rq[M - js] = ru[M - js] = o;
    }
    return;
  }
  const int mb = mbase_of(L, m);
  const bool pol = spin_polar(a, g);
  const double z = spin_arg(a, min(jn, a.npairs), pol);
  const size_t np = (size_t)(a.mmax + 1) * a.ngrp * 32, so = (size_t)m * a.ngrp * 32 + g * 32 + lane;
  const int isp = __ldg(a.ist + so), isn = __ldg(a.ist + np + so);
  const int lb = ls - ((ls + m + s) & 1);
  auto fetch = [&](int c, int buf) {
    const int l = mb + max(l0, min(c + lane, L));
    copy16(&s_t[warp][buf].ab[lane], (pol ? a.ab[1] : a.ab[0]) + l);
    copy8(&s_t[warp][buf].bm[lane], (pol ? a.bm[1] : a.bm[0]) + l);
    copy16(&s_c[warp][buf][2 * lane], ap + l);
    copy16(&s_c[warp][buf][2 * lane + 1], am + l);
    copies_commit();
  };
  double p1 = 0.0, p2 = 0.0, n1 = 0.0, n2 = 0.0;
  // north: PA = sum pv A+, NA = sum nv A-; south: D1 = sum p nv A+, D2 = sum p pv A-
  float4 PA = make_float4(0.f, 0.f, 0.f, 0.f), NA = PA, D1 = PA, D2 = PA;
  fetch(lb, 0);
  int buf = 0;
  for (int c = lb; c <= L; c += 32, buf ^= 1) {
    fetch(c + 32, buf ^ 1);
    copies_wait<1>();
    __syncwarp();
    const int nd = min(32, L - c + 1);
    auto degree = [&](int t, float sg) {
      const int l = c + t;
      const double2 ab = s_t[warp][buf].ab[t];
      const double bm = s_t[warp][buf].bm[t];
      const float4 A = s_c[warp][buf][2 * t], B = s_c[warp][buf][2 * t + 1];
      if (l == isp) {
        const double2 w = __ldg(a.st + so);
        p1 = w.x;
        p2 = w.y;
      }
      if (l == isn) {
        const double2 w = __ldg(a.st + np + so);
        n1 = w.x;
        n2 = w.y;
      }
      const double qp = fma(fma(ab.x, z, ab.y), p1, -p2), qn = fma(fma(ab.x, z, bm), n1, -n2);
      float ph, pl, nh, nl;
      split_qr(p1, ph, pl);
      split_qr(n1, nh, nl);
      p2 = p1;
      p1 = qp;
      n2 = n1;
      n1 = qn;
      cmac(PA, A, ph, pl);
      cmac(NA, B, nh, nl);
      cmac(D1, A, sg * nh, sg * nl);
      cmac(D2, B, sg * ph, sg * pl);
    };
    for (int t = 0; t < nd; t += 2) {
      degree(t, 1.f);
      if (t + 1 < nd) degree(t + 1, -1.f);
    }
    __syncwarp();
  }
  copies_wait<0>();  // the chunk past the last one
  if (jn > a.npairs) return;
  const double sgs = (s & 1) ? -1.0 : 1.0;               // (-1)^s
  const double sgd = ((m + s) & 1) ? -1.0 : 1.0;         // doubling sign (-1)^(m+s)
  const double2 pa = cval(PA), na = cval(NA), d1 = cval(D1), d2 = cval(D2);
  const double2 fqn = make_double2(pa.x + na.x, pa.y + na.y);
  const double2 fun = make_double2(pa.y - na.y, na.x - pa.x);              // -i (PA - NA)
  const double2 fqs = make_double2(sgs * (d1.x + d2.x), sgs * (d1.y + d2.y));
  const double2 fus = make_double2(sgs * (d1.y - d2.y), sgs * (d2.x - d1.x));  // (-1)^s i (D2 - D1)
  rq[jn] = fqn;
  ru[jn] = fun;
  rq[M - jn] = make_double2(sgd * fqn.x, sgd * fqn.y);
  ru[M - jn] = make_double2(sgd * fun.x, sgd * fun.y);
  if (js != jn) {
    rq[js] = fqs;
    ru[js] = fus;
    rq[M - js] = make_double2(sgd * fqs.x, sgd * fqs.y);
    ru[M - js] = make_double2(sgd * fus.x, sgd * fus.y);
  }
}

// the poles theta = 0, pi: only the order m = s is nonzero there, with
// W(0) = -X(0) = N_l / 2 and W(pi) = X(pi) = (-1)^(l+s) (-1)^s N_l / 2, N_l = sqrt((2l+1)/4pi);
// the pole entries of every other order are set to zero (the adjoint uses the
// same buffers for the theta spectra)
__global__ void spin_poles_k(int L, int mmax, int s, int M, const double2* __restrict__ glm,
                             const double2* __restrict__ clm, double2* __restrict__ GQ, double2* __restrict__ GU) {
  __shared__ double red[8][256];
  for (int m = threadIdx.x; m <= mmax; m += blockDim.x) {
    if (m == s) continue;
    GQ[(size_t)m * M] = GU[(size_t)m * M] = make_double2(0.0, 0.0);
    GQ[(size_t)m * M + M / 2] = GU[(size_t)m * M + M / 2] = make_double2(0.0, 0.0);
  }
  double v[8] = {0, 0, 0, 0, 0, 0, 0, 0};  // Q(0), U(0), Q(pi), U(pi), re and im each
  if (s <= mmax) {
    const int mb = s * (2 * L + 1 - s) / 2;
    const double sgs = (s & 1) ? -1.0 : 1.0;
    for (int l = s + threadIdx.x; l <= L; l += blockDim.x) {
      const double nl = sqrt((2.0 * l + 1.0) / (4.0 * 3.14159265358979323846));
      const double2 g = glm[mb + l], c = clm[mb + l];
      const double gi = s == 0 ? 0.0 : g.y, ci = s == 0 ? 0.0 : c.y;
      double W = 0.5 * nl, X = -0.5 * nl;
      v[0] += g.x * W - ci * X;
      v[1] += gi * W + c.x * X;
      v[2] += c.x * W + gi * X;
      v[3] += ci * W - g.x * X;
      W = X = 0.5 * nl * sgs * (((l + s) & 1) ? -1.0 : 1.0);
      v[4] += g.x * W - ci * X;
      v[5] += gi * W + c.x * X;
      v[6] += c.x * W + gi * X;
      v[7] += ci * W - g.x * X;
    }
  }
  for (int k = 0; k < 8; ++k) red[k][threadIdx.x] = v[k];
  __syncthreads();
  for (int h = blockDim.x / 2; h > 0; h >>= 1) {
    if ((int)threadIdx.x < h)
      for (int k = 0; k < 8; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0 && s <= mmax) {
    double2* rq = GQ + (size_t)s * M;
    double2* ru = GU + (size_t)s * M;
    rq[0] = make_double2(red[0][0], red[1][0]);
    ru[0] = make_double2(red[2][0], red[3][0]);
    rq[M / 2] = make_double2(red[4][0], red[5][0]);
    ru[M / 2] = make_double2(red[6][0], red[7][0]);
  }
}

// shared-memory slots of the adjoint: per warp, 4 degrees x 32 lanes x 8
// floats (G and C as float pairs); a lane's 8 floats start at a multiple of
// 12 floats (two conflict-free 16-byte stores per quarter warp) and the
// degrees 392 = 8 (mod 32) floats apart, so that the transpose read (lane t:
// degree t/4, float pair t mod 4 of one lane) hits distinct banks per half warp
constexpr int SPIN_SL = 12, SPIN_SD = 32 * SPIN_SL + 8;

// adjoint: from the theta spectra HQ, HU (inverse theta FFT done), fold with
// the spin sign, then per degree G += pv U1 + nv U2, C += i (nv V2 - pv V1)
// over the warp's ring pairs; partial rows [group][nalm] as float pairs, G in
// pg and C in pc, from the group's first degree on
__global__ void __launch_bounds__(128) spin_adj_k(SpinArgs a, const double2* __restrict__ HQ,
                                                  const double2* __restrict__ HU, float4* __restrict__ pg,
                                                  float4* __restrict__ pc, int64_t nalm) {
  __shared__ __align__(16) float slots[4][4 * SPIN_SD];
  __shared__ __align__(16) SpinChunk s_t[4][2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int it = blockIdx.x * 4 + warp;
  if (it >= (a.mmax + 1) * a.ngrp) return;
  float* sl = slots[warp];
  const int m = it / a.ngrp, g = it % a.ngrp;
  const int L = a.lmax, s = a.s, M = a.M;
  const int ls = __ldg(a.gst + it);
  if (ls > L) return;
  const int l0 = m > s ? m : s;
  const int mb = mbase_of(L, m);
  const bool pol = spin_polar(a, g);
  const double hs = (s & 1) ? -0.5 : 0.5;  // (-1)^s / 2
  const double sgd = ((m + s) & 1) ? -1.0 : 1.0;
  const double2* hq = HQ + (size_t)m * M;
  const double2* hu = HU + (size_t)m * M;
  // transpose-read role of this lane: float pair k = t mod 16 (degree k / 4,
  // component k mod 4: G re, G im, C re, C im) summed over lanes 16 h .. 16 h + 15
  const int tk = lane & 15, th = lane >> 4, td = tk >> 2, tc = tk & 3;
  const int jn = g * 32 + lane + 1;
  const bool valid = jn <= a.npairs;
  const double z = spin_arg(a, min(jn, a.npairs), pol);
  const size_t np = (size_t)(a.mmax + 1) * a.ngrp * 32, so = (size_t)m * a.ngrp * 32 + g * 32 + lane;
  const int isp = __ldg(a.ist + so), isn = __ldg(a.ist + np + so);
  // D^dagger with the spin sign: F(theta) = H(theta) + (-1)^(m+s) H(2 pi - theta)
  double2 qn = make_double2(0, 0), qs = qn, un = qn, us = qn;
  if (valid) {
    const int js = M / 2 - jn;
    qn = make_double2(hq[jn].x + sgd * hq[M - jn].x, hq[jn].y + sgd * hq[M - jn].y);
    un = make_double2(hu[jn].x + sgd * hu[M - jn].x, hu[jn].y + sgd * hu[M - jn].y);
    if (js != jn) {
      qs = make_double2(hq[js].x + sgd * hq[M - js].x, hq[js].y + sgd * hq[M - js].y);
      us = make_double2(hu[js].x + sgd * hu[M - js].x, hu[js].y + sgd * hu[M - js].y);
    }
  }
  // B+ = H^Q + i H^U, B- = H^Q - i H^U at each ring; U1 +- = (B+_n +- B-_s) / 2,
  // U2 +- = (-1)^s (B-_n +- B+_s) / 2 as float pairs
  const double2 bpn = make_double2(qn.x - un.y, qn.y + un.x), bmn = make_double2(qn.x + un.y, qn.y - un.x);
  const double2 bps = make_double2(qs.x - us.y, qs.y + us.x), bms = make_double2(qs.x + us.y, qs.y - us.x);
  float4 u1p, u1m, u2p, u2m;
  df_split(0.5 * (bpn.x + bms.x), u1p.x, u1p.y);
  df_split(0.5 * (bpn.y + bms.y), u1p.z, u1p.w);
  df_split(0.5 * (bpn.x - bms.x), u1m.x, u1m.y);
  df_split(0.5 * (bpn.y - bms.y), u1m.z, u1m.w);
  df_split(hs * (bmn.x + bps.x), u2p.x, u2p.y);
  df_split(hs * (bmn.y + bps.y), u2p.z, u2p.w);
  df_split(hs * (bmn.x - bps.x), u2m.x, u2m.y);
  df_split(hs * (bmn.y - bps.y), u2m.z, u2m.w);
  float4* og = pg + (size_t)g * nalm + mb;
  float4* oc = pc + (size_t)g * nalm + mb;
  auto fetch = [&](int c, int buf) {
    const int l = mb + max(l0, min(c + lane, L));
    copy16(&s_t[warp][buf].ab[lane], (pol ? a.ab[1] : a.ab[0]) + l);
    copy8(&s_t[warp][buf].bm[lane], (pol ? a.bm[1] : a.bm[0]) + l);
    copies_commit();
  };
  double p1 = 0.0, p2 = 0.0, n1 = 0.0, n2 = 0.0;
  const int lb = ls - ((ls + m + s) & 1);
  fetch(lb, 0);
  for (int c = lb; c <= L; c += 4) {
    const int at = c - lb, buf = (at >> 5) & 1;
    if ((at & 31) == 0) {
      fetch(c + 32, buf ^ 1);
      copies_wait<1>();
      __syncwarp();
    }
    const int nd = min(4, L - c + 1);
    // one degree; G with (x1, x2), C with (y1, y2): p and -p
    auto degree = [&](int t, const float4& x1, const float4& x2, const float4& y1, const float4& y2) {
      const int l = c + t;
      const double2 ab = s_t[warp][buf].ab[(at & 31) + t];
      const double bm = s_t[warp][buf].bm[(at & 31) + t];
      if (l == isp) {
        const double2 w = __ldg(a.st + so);
        p1 = w.x;
        p2 = w.y;
      }
      if (l == isn) {
        const double2 w = __ldg(a.st + np + so);
        n1 = w.x;
        n2 = w.y;
      }
      const double qp = fma(fma(ab.x, z, ab.y), p1, -p2), qn1 = fma(fma(ab.x, z, bm), n1, -n2);
      float ph, pl, nh, nl;
      split_qr(p1, ph, pl);
      split_qr(n1, nh, nl);
      p2 = p1;
      p1 = qp;
      n2 = n1;
      n1 = qn1;
      float4 gv, w;
      cprod(gv, x1, ph, pl);
      cmac_open(gv, x2, nh, nl);
      cprod(w, y2, nh, nl);
      cmac_open(w, y1, -ph, -pl);
      // C = i w = (-w.im, w.re)
      float4* dst = reinterpret_cast<float4*>(sl + t * SPIN_SD + lane * SPIN_SL);
      dst[0] = gv;
      dst[1] = make_float4(-w.z, -w.w, w.x, w.y);
    };
#pragma unroll 1
    for (int t = 0; t < nd; t += 2) {
      degree(t, u1p, u2p, u1m, u2m);  // l + m + s even: p = 1
      if (t + 1 < nd) degree(t + 1, u1m, u2m, u1p, u2p);
    }
    __syncwarp();
    const float* src = sl + td * SPIN_SD + (16 * th) * SPIN_SL + 2 * tc;
    float sh = 0.f, slo = 0.f;
    if (td < nd) {
#pragma unroll 4
      for (int i = 0; i < 16; ++i) {
        const float2 v = *reinterpret_cast<const float2*>(src + i * SPIN_SL);
        df_add(sh, slo, v.x, v.y);
      }
    }
    const float oh = __shfl_xor_sync(FULL, sh, 16), ol = __shfl_xor_sync(FULL, slo, 16);
    df_add(sh, slo, oh, ol);
    if (th == 0 && td < nd && c + td >= ls) {
      float4* row = tc < 2 ? og : oc;
      reinterpret_cast<float2*>(row + c + td)[tc & 1] = make_float2(sh, slo);
    }
    __syncwarp();
  }
  copies_wait<0>();  // the chunk past the last one
}

// c_lm = s_l times the sum over the partial rows of the groups that have
// started at degree l, in a fixed order (float pairs), plus the poles (order
// s); entries with l < s are 0, Im of the m = 0 entries is 0
__global__ void spin_adj_reduce_k(const float4* __restrict__ pg, const float4* __restrict__ pc,
                                  const int* __restrict__ gst, const double* __restrict__ scl, int nrows,
                                  int64_t nalm, int L, int mmax, int s, int M, const double2* __restrict__ HQ,
                                  const double2* __restrict__ HU, double2* __restrict__ og,
                                  double2* __restrict__ oc) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nalm) return;
  // (l, m) of packed index i: order m holds l = m..L at m (2L + 1 - m) / 2 + l,
  // so m is the largest order whose first entry m (2L + 1 - m) / 2 + m is <= i
  int lo = 0, hi = mmax;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if ((int64_t)mid * (2 * L + 1 - mid) / 2 + mid <= i)
      lo = mid;
    else
      hi = mid - 1;
  }
  const int m = lo;
  const int l = (int)(i - (int64_t)m * (2 * L + 1 - m) / 2);
  double g0 = 0, g1 = 0, c0 = 0, c1 = 0;
  if (l >= s) {
    float4 sg = make_float4(0.f, 0.f, 0.f, 0.f), sc = sg;
    for (int r = 0; r < nrows; ++r) {
      if (l < __ldg(gst + m * nrows + r)) continue;
      const float4 a = pg[(size_t)r * nalm + i], b = pc[(size_t)r * nalm + i];
      df_add(sg.x, sg.y, a.x, a.y);
      df_add(sg.z, sg.w, a.z, a.w);
      df_add(sc.x, sc.y, b.x, b.y);
      df_add(sc.z, sc.w, b.z, b.w);
    }
    const double f = scl[i];
    g0 = f * df_value(sg.x, sg.y);
    g1 = f * df_value(sg.z, sg.w);
    c0 = f * df_value(sc.x, sc.y);
    c1 = f * df_value(sc.z, sc.w);
    if (m == s) {
      // poles: F^Q, F^U at theta = 0 (index 0) and theta = pi (index M / 2),
      // each taken once (no fold partner)
      const double nl = sqrt((2.0 * l + 1.0) / (4.0 * 3.14159265358979323846));
      const double sgs = (s & 1) ? -1.0 : 1.0;
      const double2 q0 = HQ[(size_t)m * M], u0 = HU[(size_t)m * M];
      const double2 qp = HQ[(size_t)m * M + M / 2], up = HU[(size_t)m * M + M / 2];
      double W = 0.5 * nl, X = -0.5 * nl;
      g0 += W * q0.x - X * u0.y;
      g1 += W * q0.y + X * u0.x;
      c0 += W * u0.x + X * q0.y;
      c1 += W * u0.y - X * q0.x;
      W = X = 0.5 * nl * sgs * (((l + s) & 1) ? -1.0 : 1.0);
      g0 += W * qp.x - X * up.y;
      g1 += W * qp.y + X * up.x;
      c0 += W * up.x + X * qp.y;
      c1 += W * up.y - X * qp.x;
    }
  }
  if (m == 0) g1 = c1 = 0.0;
  og[i] = make_double2(g0, g1);
  oc[i] = make_double2(c0, c1);
}

// value = p * 2^e
struct XN {
  double p;
  int e;
};
XN xn(double p, int e) {
  XN r{0.0, 0};
  if (p == 0.0) return r;
  int k;
  r.p = std::frexp(p, &k);
  r.e = e + k;
  return r;
}

SpinArgs spin_args(nusht_plan_t p) {
  SpinArgs a;
  a.lmax = p->lmax;
  a.mmax = p->mmax;
  a.M = p->sz.M;
  a.npairs = p->leg.npairs;
  a.ngrp = p->spin.nrows;
  a.s = p->opts.spin;
  a.ab[0] = p->spin.abx;
  a.ab[1] = p->spin.abs;
  a.bm[0] = p->spin.bmx;
  a.bm[1] = p->spin.bms;
  a.gst = p->spin.gst;
  a.ist = p->spin.ist;
  a.st = p->spin.st;
  return a;
}

}  // namespace

// plan time: recurrence tables, start values, ring maps and partial rows
int spin_setup(nusht_plan_t p, cudaStream_t s) {
  const int L = p->lmax, mmax = p->mmax, sp = p->opts.spin;
  const int64_t nalm = p->nalm;
  std::vector<double> mant(2 * (mmax + 1), 0.0);
  std::vector<int> ex(2 * (mmax + 1), 0), ab(2 * (mmax + 1), 0);
  const double sgs = (sp & 1) ? -1.0 : 1.0;
  for (int m = 0; m <= mmax; ++m) {
    const int l0 = std::max(m, sp);
    // start values at l0: (-1)^s sqrt((2 l0 + 1)/(4 pi)) d^l0_{m, mp} for mp = -s (lambda+), +s (lambda-)
    for (int sign = 0; sign < 2; ++sign) {
      const int mpv = sign == 0 ? -sp : sp;
      int k, a, b;
      bool neg;
      if (m >= sp) {  // d^l0_{l0, mp} = (-1)^(l0 - mp) sqrt(C(2 l0, l0 + mp)) c^(l0 + mp) s^(l0 - mp)
        k = l0 + mpv;
        a = l0 + mpv;
        b = l0 - mpv;
        neg = ((l0 - mpv) & 1) != 0;
      } else if (mpv > 0) {  // d^l0_{m, l0} = sqrt(C(2 l0, l0 + m)) c^(l0 + m) s^(l0 - m)
        k = l0 + m;
        a = l0 + m;
        b = l0 - m;
        neg = false;
      } else {  // d^l0_{m, -l0} = (-1)^(l0 + m) sqrt(C(2 l0, l0 - m)) c^(l0 - m) s^(l0 + m)
        k = l0 - m;
        a = l0 - m;
        b = l0 + m;
        neg = ((l0 + m) & 1) != 0;
      }
      XN r = xn(1.0, 0);
      for (int i = 1; i <= k; ++i) r = xn(r.p * ((double)(2 * l0 - k + i) / (double)i), r.e);
      if (r.e & 1) {
        r.p *= 2.0;
        r.e -= 1;
      }
      r = xn(std::sqrt(r.p) * std::sqrt((2.0 * l0 + 1.0) / (4.0 * M_PI)) * sgs * (neg ? -1.0 : 1.0), r.e / 2);
      mant[2 * m + sign] = r.p;
      ex[2 * m + sign] = r.e;
      ab[2 * m + sign] = (a << 16) | b;
    }
  }
  SpinTables& t = p->spin;
  t.nrows = (p->leg.npairs + 31) / 32;
  const size_t groups = (size_t)(mmax + 1) * t.nrows, np = groups * 32;
  NUSHT_TRY(dev_alloc((void**)&t.abx, nalm * 16, &p->bytes));
  NUSHT_TRY(dev_alloc((void**)&t.abs, nalm * 16, &p->bytes));
  NUSHT_TRY(dev_alloc((void**)&t.bmx, nalm * 8, &p->bytes));
  NUSHT_TRY(dev_alloc((void**)&t.bms, nalm * 8, &p->bytes));
  NUSHT_TRY(dev_alloc((void**)&t.sc, nalm * 8, &p->bytes));
  NUSHT_TRY(dev_alloc((void**)&t.gst, groups * 4, &p->bytes));
  NUSHT_TRY(dev_alloc((void**)&t.ist, 2 * np * 4, &p->bytes));
  NUSHT_TRY(dev_alloc((void**)&t.st, 2 * np * 16, &p->bytes));
  // start values of the chains, used by the set-up only
  const size_t mb8 = mant.size() * 8, mb4 = ex.size() * 4;
  char* tmp = nullptr;
  NUSHT_TRY(dev_alloc((void**)&tmp, mb8 + 2 * mb4, nullptr));
  cudaError_t e = cudaMemcpy(tmp, mant.data(), mb8, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(tmp + mb8, ex.data(), mb4, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(tmp + mb8 + mb4, ab.data(), mb4, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemsetAsync(t.sc, 0, nalm * 8, s);
  if (e == cudaSuccess) {
    spin_tab_k<<<(mmax + 4) / 4, 128, 0, s>>>(L, mmax, sp, t.abx, t.bmx, t.abs, t.bms, t.sc);
    spin_start_k<<<(int)((groups + 3) / 4), 128, 0, s>>>(spin_args(p), (const double*)tmp, (const int*)(tmp + mb8),
                                                         (const int*)(tmp + mb8 + mb4), t.gst, t.ist, t.st);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  dev_free(tmp);
  if (e != cudaSuccess) return cuda_status(e, "spin tables");
  const size_t gbytes = (size_t)(mmax + 1) * p->sz.M * sizeof(double2);
  NUSHT_TRY(dev_alloc((void**)&t.GQ, gbytes, &p->bytes));
  NUSHT_TRY(dev_alloc((void**)&t.GU, gbytes, &p->bytes));
  NUSHT_CUDA(cudaMemsetAsync(t.GQ, 0, gbytes, s));
  NUSHT_CUDA(cudaMemsetAsync(t.GU, 0, gbytes, s));
  NUSHT_TRY(dev_alloc((void**)&t.ap, nalm * sizeof(float4), &p->bytes));
  NUSHT_TRY(dev_alloc((void**)&t.am, nalm * sizeof(float4), &p->bytes));
  const size_t pbytes = (size_t)t.nrows * nalm * sizeof(float4);
  NUSHT_TRY(dev_alloc((void**)&t.pg, pbytes, &p->bytes));
  NUSHT_TRY(dev_alloc((void**)&t.pc, pbytes, &p->bytes));
  NUSHT_CUDA(cudaStreamSynchronize(s));
  return NUSHT_OK;
}

void spin_free(nusht_plan_t p) {
  SpinTables& t = p->spin;
  for (void* q : {(void*)t.abx, (void*)t.abs, (void*)t.bmx, (void*)t.bms, (void*)t.sc, (void*)t.gst, (void*)t.ist,
                  (void*)t.st, (void*)t.GQ, (void*)t.GU, (void*)t.ap, (void*)t.am, (void*)t.pg, (void*)t.pc})
    dev_free(q);
  t = SpinTables();
}

int spin_legendre_synth(nusht_plan_t p, const void* glm, const void* clm, cudaStream_t s) {
  const SpinArgs a = spin_args(p);
  const int nitems = (p->mmax + 1) * a.ngrp;
  spin_scale_k<<<(int)((p->nalm + 255) / 256), 256, 0, s>>>((const double2*)glm, (const double2*)clm, p->spin.sc,
                                                             p->nalm, p->lmax, p->opts.spin, p->spin.ap, p->spin.am);
  spin_synth_k<<<(nitems + 3) / 4, 128, 0, s>>>(a, p->spin.ap, p->spin.am, p->spin.GQ, p->spin.GU);
  spin_poles_k<<<1, 256, 0, s>>>(p->lmax, p->mmax, p->opts.spin, p->sz.M, (const double2*)glm, (const double2*)clm,
                                 p->spin.GQ, p->spin.GU);
  NUSHT_CUDA(cudaGetLastError());
  return NUSHT_OK;
}

int spin_legendre_adjoint(nusht_plan_t p, void* glm, void* clm, cudaStream_t s) {
  const SpinArgs a = spin_args(p);
  const int nitems = (p->mmax + 1) * a.ngrp;
  spin_adj_k<<<(nitems + 3) / 4, 128, 0, s>>>(a, p->spin.GQ, p->spin.GU, p->spin.pg, p->spin.pc, p->nalm);
  spin_adj_reduce_k<<<(int)((p->nalm + 255) / 256), 256, 0, s>>>(p->spin.pg, p->spin.pc, p->spin.gst, p->spin.sc,
                                                                 p->spin.nrows, p->nalm,
                                                                 p->lmax, p->mmax, p->opts.spin, p->sz.M,
                                                                 p->spin.GQ, p->spin.GU, (double2*)glm,
                                                                 (double2*)clm);
  NUSHT_CUDA(cudaGetLastError());
  return NUSHT_OK;
}

}  // namespace nusht
