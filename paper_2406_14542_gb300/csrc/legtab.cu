// legtab.cu -- the iso-latitude step S and its adjoint of mixed plans from a
// recurrence table.
//
// The recurrence values at the rings do not depend on the coefficients: the
// plan runs the FP64 recurrence of legendre.cu once (q_l = Pbar_l / Ahat_l) and
// keeps the values as floats in HBM; a call streams them through FP32 sums, so
// the stream is the cost.  Per (order m, group of 32 ring pairs) the table
// begins at the first step i (degrees m + 2i and m + 2i + 1) with a nonzero
// float, and the even and odd degrees are two streams of chunks: one float4
// per lane (ring pair) holds four steps.
//
// Synthesis reads both streams; its sums are those of the per-call recurrence
// (legendre_synth_k<float>) term by term, bit for bit.  The adjoint reads only
// the odd stream wherever cos(theta) >= TAB_XMIN: with l odd in this sense and
// eps_l^2 = (l^2 - m^2) / (4 l^2 - 1),
//   Pbar_{l-1} = eps_l Pbar_l / x + eps_{l-1} Pbar_{l-2} / x,
// so the even coefficients follow from sums of the odd values against S / x
// (as in legendre2.cu).  There 1 / x <= 4 multiplies the rounding of a value
// (1.6 in the mean square over the rings), far below the error of the FP32
// sums; the blocks of 128 pairs nearer the equator read both streams.  (Half
// a table would serve the synthesis as well, 0.63 ms instead of 0.95 at lmax
// 2047, but not with the same bits, which the position gradients of mixed
// plans, given in double, are held to.)
//
// Measured against one stream of every degree per kept block of 128 pairs,
// lmax 2047: synthesis 1.18 -> 0.95 ms (6.4 GB at 6.7 TB/s, the copy
// bandwidth), adjoint with its reduction 1.42 -> 0.85 ms (3.9 GB; shuffles and
// strided reads hold it to about 0.77 of the copy bandwidth).
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <type_traits>
#include <vector>

#include "dfloat.cuh"
#include "nusht_internal.cuh"
#include "recurrence.cuh"

namespace nusht {

namespace {

using namespace rec;
constexpr unsigned FULL = 0xffffffffu;

struct TabArgs {
  int lmax, mmax, M, npairs, ngrp;
  const double* c;
  const int8_t* dshift;
  const double* cm;
  const double* ring_x;
  const double* ring_s;
  const float4* tab;
  const int64_t* off;  // [order][group]: first chunk of the even stream, in chunks of 32 float4
  const int* gst;      // [order][group]: first step (INT_MAX: none)
  int nA;
};
__device__ __forceinline__ int chunks_of(int n, int gs) { return (n + 3) / 4 - (gs >> 2); }

// the recurrence value as the table holds it
__device__ __forceinline__ float tab_value(const Chain& ch) {
  return ch.valid && ch.E == 0 ? to_f32(ch.q1) : 0.f;
}
// q_l of one degree more than the tables reach (the last step's odd degree is
// lmax + 1 where lmax - m is even): same segment, the rational c_l
__device__ __forceinline__ void tab_step(const TabArgs& a, Chain& ch, int mb, int l, int m) {
  if (l <= a.lmax) {
    chain_step(ch, __ldg(a.c + mb + l), __ldg(a.dshift + mb + l));
  } else {
    const double dl = l, dm = m;
    chain_step(ch, l == m + 1 ? 0.0 : ((dl - 1.0 - dm) * (dl - 1.0 + dm)) / ((2.0 * dl - 3.0) * (2.0 * dl - 1.0)), 0);
  }
}

// plan time, one warp per (order, group): the first step with a nonzero value,
// or (tab given) the streams from it
__global__ void __launch_bounds__(128) tab_build_k(TabArgs a, int* __restrict__ gst, float4* __restrict__ tab) {
  const int lane = threadIdx.x & 31;
  const int it = blockIdx.x * 4 + (threadIdx.x >> 5);
  if (it >= (a.mmax + 1) * a.ngrp) return;
  const int m = it / a.ngrp, g = it % a.ngrp, n = steps_of(a.lmax, m), mb = mbase_of(a.lmax, m);
  Chain ch;
  chain_init(ch, a, m, g * 32 + lane + 1);
  if (!tab) {
    int first = INT_MAX;
    for (int i = 0; i < n && first == INT_MAX; ++i) {
      float v = fabsf(tab_value(ch));
      tab_step(a, ch, mb, m + 2 * i + 1, m);
      v += fabsf(tab_value(ch));
      if (__any_sync(FULL, v != 0.f)) first = i;
      if (i + 1 < n) tab_step(a, ch, mb, m + 2 * i + 2, m);
    }
    if (lane == 0) gst[it] = first;
    return;
  }
  const int gs = a.gst[it];
  if (gs >= n) return;
  const int nc = chunks_of(n, gs), c0 = gs >> 2;
  float4* out = tab + a.off[it] * 32 + lane;
  float4 e, o;
  for (int i = 0; i < 4 * ((n + 3) / 4); ++i) {
    float ve = 0.f, vo = 0.f;
    if (i < n) {
      ve = tab_value(ch);
      tab_step(a, ch, mb, m + 2 * i + 1, m);
      vo = tab_value(ch);
      if (i + 1 < n) tab_step(a, ch, mb, m + 2 * i + 2, m);
    }
    const int k = i & 3;
    if (k == 0) e.x = ve, o.x = vo;
    if (k == 1) e.y = ve, o.y = vo;
    if (k == 2) e.z = ve, o.z = vo;
    if (k == 3) e.w = ve, o.w = vo;
    const int c = (i >> 2) - c0;
    if (k == 3 && c >= 0) {
      out[(size_t)c * 32] = e;
      out[(size_t)(nc + c) * 32] = o;
    }
  }
}

// plan time: the factors of the odd sums, per step (l = m + 2i + 1)
__global__ void __launch_bounds__(256) tab_scale_k(int L, const double* __restrict__ ahat, double* __restrict__ sc,
                                                   double* __restrict__ w1, double* __restrict__ w2) {
  const int m = blockIdx.y, i = blockIdx.x * 256 + threadIdx.x;
  if (i >= steps_of(L, m)) return;
  const int l = m + 2 * i + 1;
  const double m2 = (double)m * m;
  auto eps2 = [&](double d) { return (d * d - m2) / (4.0 * d * d - 1.0); };
  const double* ah = ahat + mbase_of(L, m);
  // Ahat_l = Ahat_{l-1} / eps_l inside a segment
  const double s = l <= L ? ah[l] : ah[l - 1] / sqrt(eps2(l));
  const int64_t k = base_of(L, m) + i;
  sc[k] = s;
  w1[k] = s * sqrt(eps2(l));
  w2[k] = s * sqrt(eps2(l + 1.0));
}

// per call: a_l Ahat_l of a step's two degrees as float, and the poles
__global__ void __launch_bounds__(256) tab_coef_k(const float2* __restrict__ alm, int L, int mmax, int M,
                                                  const double* __restrict__ ahat,
                                                  const double* __restrict__ pole_norm, float4* __restrict__ ao,
                                                  float2* __restrict__ G) {
  const int m = blockIdx.y;
  if (m > mmax) {
    if (blockIdx.x) return;
    __shared__ double sn[256], ss[256];
    double nn = 0.0, sp = 0.0;
    for (int l = threadIdx.x; l <= L; l += 256) {
      const double v = (double)alm[l].x * pole_norm[l];
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
      G[0] = make_float2((float)sn[0], 0.f);
      G[M / 2] = make_float2((float)ss[0], 0.f);
    }
    return;
  }
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= steps_of(L, m)) return;
  const int l = m + 2 * i, mb = mbase_of(L, m);
  const float2 e = alm[mb + l], o = l < L ? alm[mb + l + 1] : make_float2(0.f, 0.f);
  const double fe = ahat[mb + l], fo = l < L ? ahat[mb + l + 1] : 0.0;
  float4 r = make_float4((float)(e.x * fe), (float)(e.y * fe), (float)(o.x * fo), (float)(o.y * fo));
  if (m == 0) r.y = r.w = 0.f;  // Im(a_l0) is ignored
  ao[base_of(L, m) + i] = r;
}

// synthesis: one warp per (order, group)
__global__ void __launch_bounds__(128) tab_synth_k(TabArgs a, const int* __restrict__ items, int nitems,
                                                   const float4* __restrict__ ao, float2* __restrict__ G) {
  const int lane = threadIdx.x & 31;
  const int it = blockIdx.x * 4 + (threadIdx.x >> 5);
  if (it >= nitems) return;
  const int v = __ldg(items + it);
  const int m = v >> 16, g = v & 0xffff, n = steps_of(a.lmax, m), gi = m * a.ngrp + g;
  const int c0 = __ldg(a.gst + gi) >> 2, nc = (n + 3) / 4;
  const float4* qe = a.tab + __ldg(a.off + gi) * 32 + lane;
  const float4* qo = qe + (size_t)(nc - c0) * 32;
  const float4* cf = ao + base_of(a.lmax, m);
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);  // (re, im) of the even and the odd sum
  auto add = [&](int i, float pe, float po) {
    const float4 c = __ldg(cf + min(i, n - 1));  // steps past the last have values 0
    s.x = fmaf(c.x, pe, s.x);
    s.y = fmaf(c.y, pe, s.y);
    s.z = fmaf(c.z, po, s.z);
    s.w = fmaf(c.w, po, s.w);
  };
  auto chunk = [&](int c, const float4 e, const float4 o) {
    add(4 * c, e.x, o.x);
    add(4 * c + 1, e.y, o.y);
    add(4 * c + 2, e.z, o.z);
    add(4 * c + 3, e.w, o.w);
  };
  int c = c0;
  for (; c + 2 <= nc; c += 2, qe += 64, qo += 64) {
    const float4 e0 = __ldcs(qe), o0 = __ldcs(qo), e1 = __ldcs(qe + 32), o1 = __ldcs(qo + 32);
    chunk(c, e0, o0);
    chunk(c + 1, e1, o1);
  }
  if (c < nc) chunk(c, __ldcs(qe), __ldcs(qo));
  const int jn = g * 32 + lane + 1;
  if (jn > a.npairs) return;
  const int M = a.M, js = M / 2 - jn;
  const double sg = (m & 1) ? -1.0 : 1.0;
  const double er = s.x, ei = s.y, orr = s.z, oi = s.w;
  float2* row = G + (size_t)m * M;
  row[jn] = make_float2((float)(er + orr), (float)(ei + oi));
  row[M - jn] = make_float2((float)(sg * (er + orr)), (float)(sg * (ei + oi)));
  if (js != jn) {
    row[js] = make_float2((float)(er - orr), (float)(ei - oi));
    row[M - js] = make_float2((float)(sg * (er - orr)), (float)(sg * (ei - oi)));
  }
}

// Sums of N values per lane over the warp: N / 2 exchanges, then fewer; lane
// bits 4, 3, ... select the value a lane ends with
template <int N>
__device__ __forceinline__ float scatter_sum(float (&v)[N], int lane) {
  int o = 16;
#pragma unroll
  for (int n = N / 2; n >= 1; n /= 2, o /= 2) {
    const bool up = lane & o;
#pragma unroll
    for (int k = 0; k < n; ++k) {
      const float send = up ? v[k] : v[k + n], keep = up ? v[k + n] : v[k];
      v[k] = keep + __shfl_xor_sync(FULL, send, o);
    }
  }
  for (; o >= 1; o /= 2) v[0] += __shfl_xor_sync(FULL, v[0], o);
  return v[0];
}

// adjoint: one warp per (order, block of 128 pairs), four groups per lane so
// that the reduction over the lanes is shared; partial[block][step] as
// (even re, im, odd re, im), the even part against S / x in polar blocks
__global__ void __launch_bounds__(128) tab_adj_k(TabArgs a, const int* __restrict__ items, int nitems,
                                                 const float2* __restrict__ Gt, float4* __restrict__ partial,
                                                 int64_t n2) {
  const int lane = threadIdx.x & 31;
  const int it = blockIdx.x * 4 + (threadIdx.x >> 5);
  if (it >= nitems) return;
  const int v = __ldg(items + it);
  const int m = v >> 16, blk = v & 0xffff, n = steps_of(a.lmax, m), M = a.M, nc = (n + 3) / 4;
  const bool A = blk < a.nA;
  const float sg = (m & 1) ? -1.f : 1.f;
  const float2* row = Gt + (size_t)m * M;
  const float4* q[4];  // the odd stream; the even one lies nc - c0 chunks before it
  int c0[4], cm = INT_MAX;
  float2 SE[4], SO[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int g = blk * 4 + k, gi = m * a.ngrp + g;
    const int gs = g < a.ngrp ? __ldg(a.gst + gi) : INT_MAX;
    c0[k] = gs < n ? gs >> 2 : INT_MAX;
    cm = min(cm, c0[k]);
    q[k] = gs < n ? a.tab + (__ldg(a.off + gi) + nc - c0[k]) * 32 + lane : nullptr;
    const int jn = g * 32 + lane + 1;
    float2 fn = make_float2(0.f, 0.f), fs = fn;
    float ix = 1.f;
    if (gs < n && jn <= a.npairs) {
      const int js = M / 2 - jn;
      const float2 u0 = row[jn], u1 = row[M - jn];
      fn = make_float2(u0.x + sg * u1.x, u0.y + sg * u1.y);
      if (js != jn) {
        const float2 h0 = row[js], h1 = row[M - js];
        fs = make_float2(h0.x + sg * h1.x, h0.y + sg * h1.y);
      }
      if (A) ix = 1.f / (float)__ldg(a.ring_x + jn - 1);
    }
    SE[k] = make_float2(ix * (fn.x + fs.x), ix * (fn.y + fs.y));
    SO[k] = make_float2(fn.x - fs.x, fn.y - fs.y);
  }
  float* out = reinterpret_cast<float*>(partial + (size_t)blk * n2 + base_of(a.lmax, m));
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  float4 o[4], on[4], e[4], en[4];
  auto load = [&](int c, float4 (&po)[4], float4 (&pe)[4]) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const bool in = c >= c0[k] && c < nc;
      po[k] = in ? __ldcs(q[k] + (size_t)(c - c0[k]) * 32) : zero;
      if (!A) pe[k] = in ? __ldcs(q[k] - (size_t)(nc - c) * 32) : zero;
    }
  };
  load(cm, o, e);
  for (int c = cm; c < nc; ++c) {
    load(c + 1, on, en);
    float s[16];
#pragma unroll
    for (int t = 0; t < 16; ++t) s[t] = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float4 pe = A ? o[k] : e[k];
      const float we[4] = {pe.x, pe.y, pe.z, pe.w}, wo[4] = {o[k].x, o[k].y, o[k].z, o[k].w};
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        s[4 * t] = fmaf(we[t], SE[k].x, s[4 * t]);
        s[4 * t + 1] = fmaf(we[t], SE[k].y, s[4 * t + 1]);
        s[4 * t + 2] = fmaf(wo[t], SO[k].x, s[4 * t + 2]);
        s[4 * t + 3] = fmaf(wo[t], SO[k].y, s[4 * t + 3]);
      }
    }
    const float r = scatter_sum(s, lane);
    const int t = lane >> 1;  // step 4 c + t / 4, component t mod 4
    if (!(lane & 1) && 4 * c + (t >> 2) < n) out[16 * (size_t)c + t] = r;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      o[k] = on[k];
      e[k] = en[k];
    }
  }
}

// c_lm from the block partials (summed as float pairs, in a fixed order): odd
// degrees Ahat_l times their sums, even ones from the odd sums against S / x of
// the polar blocks and, times their own Ahat, from the sums of the others
__global__ void __launch_bounds__(256) tab_reduce_k(TabArgs a, int nblk, const float4* __restrict__ partial,
                                                    int64_t n2, const double* __restrict__ ahat,
                                                    const double* __restrict__ sc, const double* __restrict__ w1,
                                                    const double* __restrict__ w2,
                                                    const double* __restrict__ pole_norm,
                                                    const float2* __restrict__ Gt, double wpos,
                                                    float2* __restrict__ out) {
  __shared__ double2 ev[257];
  __shared__ int start[64];  // first written step of each block (at most 64: lmax <= 16383)
  const int m = blockIdx.y, L = a.lmax, n = steps_of(L, m);
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (blockIdx.x * 256 >= n) return;
  const int64_t b0 = base_of(L, m);
  if ((int)threadIdx.x < nblk) {
    int s = INT_MAX;
    for (int k = threadIdx.x * 4; k < min((int)threadIdx.x * 4 + 4, a.ngrp); ++k) {
      const int g = __ldg(a.gst + m * a.ngrp + k);
      if (g < n) s = min(s, g & ~3);
    }
    start[threadIdx.x] = s;
  }
  __syncthreads();
  // float-pair sums over blocks [lo, hi) that have started at step s
  auto sums = [&](int s, int lo, int hi, double2* even, double2* odd) {
    float4 h = make_float4(0.f, 0.f, 0.f, 0.f), l = h;
    for (int b = lo; b < hi; ++b) {
      if (s < start[b]) continue;
      const float4 x = partial[(size_t)b * n2 + b0 + s];
      df_add(h.x, l.x, x.x, 0.f);
      df_add(h.y, l.y, x.y, 0.f);
      df_add(h.z, l.z, x.z, 0.f);
      df_add(h.w, l.w, x.w, 0.f);
    }
    *even = make_double2(df_value(h.x, l.x), df_value(h.y, l.y));
    if (odd) *odd = make_double2(df_value(h.z, l.z), df_value(h.w, l.w));
  };
  const double2 zero = make_double2(0.0, 0.0);
  double2 de = zero, od = zero, xe = zero, xo = zero;
  const int nA = min(a.nA, nblk);
  if (i < n) {
    sums(i, 0, nA, &de, &od);
    sums(i, nA, nblk, &xe, &xo);
  }
  ev[threadIdx.x + 1] = de;
  if (threadIdx.x == 0) {
    double2 h = zero;
    if (i > 0) sums(i - 1, 0, nA, &h, nullptr);
    ev[0] = h;
  }
  __syncthreads();
  if (i >= n) return;
  const int64_t k = b0 + i;
  const double2 dp = ev[threadIdx.x];
  const double f0 = w1[k], f1 = i > 0 ? w2[k - 1] : 0.0, f = sc[k];
  const int l = m + 2 * i;
  const double fe = ahat[mbase_of(L, m) + l];
  double2 ce = make_double2(fma(f0, de.x, fma(f1, dp.x, fe * xe.x)), fma(f0, de.y, fma(f1, dp.y, fe * xe.y)));
  double2 co = make_double2(f * (od.x + xo.x), f * (od.y + xo.y));
  float2* row = out + mbase_of(L, m);
  if (m == 0) {  // real
    const double np = Gt[0].x, sp = Gt[a.M / 2].x;
    ce = make_double2(ce.x + pole_norm[l] * (np + sp), 0.0);
    if (l + 1 <= L) co = make_double2(co.x + pole_norm[l + 1] * (np - sp), 0.0);
  } else {
    ce = make_double2(wpos * ce.x, wpos * ce.y);
    co = make_double2(wpos * co.x, wpos * co.y);
  }
  row[l] = make_float2((float)ce.x, (float)ce.y);
  if (l + 1 <= L) row[l + 1] = make_float2((float)co.x, (float)co.y);
}

TabArgs args_of(nusht_plan_t p) {
  TabArgs a;
  a.lmax = p->lmax;
  a.mmax = p->mmax;
  a.M = p->sz.M;
  a.npairs = p->leg.npairs;
  a.ngrp = (a.npairs + 31) / 32;
  a.c = p->leg.c;
  a.dshift = p->leg.dshift;
  a.cm = p->leg.cm;
  a.ring_x = p->leg.ring_x;
  a.ring_s = p->leg.ring_s;
  a.tab = p->tab.tab;
  a.off = p->tab.off;
  a.gst = p->tab.gst;
  a.nA = p->tab.nA;
  return a;
}

}  // namespace

// Needs the tables of legendre_build_tables.
int legtab_setup(nusht_plan_t p, cudaStream_t s) {
  LegTab& t = p->tab;
  const int L = p->lmax, mmax = p->mmax, npairs = p->leg.npairs, ngrp = (npairs + 31) / 32, M = p->sz.M;
  const size_t groups = (size_t)(mmax + 1) * ngrp, n2 = (size_t)base_of(L, mmax + 1);
  char* at = nullptr;
  auto carve = [&](auto*& q, size_t n) {
    q = reinterpret_cast<std::remove_reference_t<decltype(q)>>(at);
    at += (n * sizeof(*q) + 255) / 256 * 256;
  };
  auto layout = [&]() {
    carve(t.sc, n2);
    carve(t.w1, n2);
    carve(t.w2, n2);
    carve(t.ao, n2);
    carve(t.off, groups);
    carve(t.gst, groups);
    carve(t.items_s, groups);
    carve(t.items_a, groups);
  };
  layout();
  const size_t slab = (size_t)at;
  NUSHT_TRY(dev_alloc(&t.slab, slab, &p->bytes));
  at = (char*)t.slab;
  layout();
  t.n2 = (int64_t)n2;
  t.nA = 0;
  while ((t.nA + 1) * 128 <= npairs && std::cos(2.0 * M_PI * (t.nA + 1) * 128 / M) >= TAB_XMIN) ++t.nA;
  const int nb = (int)((groups + 3) / 4);
  tab_build_k<<<nb, 128, 0, s>>>(args_of(p), t.gst, nullptr);
  tab_scale_k<<<dim3((steps_of(L, 0) + 255) / 256, mmax + 1), 256, 0, s>>>(L, p->leg.ahat, t.sc, t.w1, t.w2);
  NUSHT_CUDA(cudaGetLastError());
  std::vector<int> gst(groups), is, ia;
  NUSHT_CUDA(cudaMemcpyAsync(gst.data(), t.gst, groups * 4, cudaMemcpyDeviceToHost, s));
  NUSHT_CUDA(cudaStreamSynchronize(s));
  std::vector<int64_t> off(groups, 0);
  int64_t tot = 0;
  for (int m = 0; m <= mmax; ++m)
    for (int g = 0; g < ngrp; ++g) {
      const size_t k = (size_t)m * ngrp + g;
      const int n = steps_of(L, m);
      off[k] = tot;
      if (gst[k] >= n) continue;
      tot += 2 * ((n + 3) / 4 - (gst[k] >> 2));
      is.push_back((m << 16) | g);
      if (ia.empty() || ia.back() != ((m << 16) | (g >> 2))) ia.push_back((m << 16) | (g >> 2));
    }
  const size_t need = (size_t)tot * 32 * sizeof(float4);
  size_t freeb = 0, totalb = 0;
  cudaMemGetInfo(&freeb, &totalb);
  if (need == 0 || need >= freeb / 2) {
    legtab_free(p);
    p->bytes -= slab;
    return NUSHT_OK;
  }
  t.nis = (int)is.size();
  t.nia = (int)ia.size();
  NUSHT_CUDA(cudaMemcpyAsync(t.off, off.data(), groups * 8, cudaMemcpyHostToDevice, s));
  NUSHT_CUDA(cudaMemcpyAsync(t.items_s, is.data(), is.size() * 4, cudaMemcpyHostToDevice, s));
  NUSHT_CUDA(cudaMemcpyAsync(t.items_a, ia.data(), ia.size() * 4, cudaMemcpyHostToDevice, s));
  NUSHT_TRY(dev_alloc((void**)&t.tab, need, &p->bytes));
  tab_build_k<<<nb, 128, 0, s>>>(args_of(p), t.gst, t.tab);
  NUSHT_CUDA(cudaGetLastError());
  NUSHT_CUDA(cudaStreamSynchronize(s));
  p->leg.tab_bytes = need;
  return NUSHT_OK;
}

void legtab_free(nusht_plan_t p) {
  dev_free(p->tab.tab);
  dev_free(p->tab.slab);
  p->tab = LegTab();
}

size_t legtab_partial_bytes(nusht_plan_t p) {
  return (size_t)((p->leg.npairs + 127) / 128) * (size_t)p->tab.n2 * sizeof(float4);
}

int legtab_synth(nusht_plan_t p, const void* d_alm, cudaStream_t s) {
  const LegTab& t = p->tab;
  const TabArgs a = args_of(p);
  const dim3 cg((steps_of(p->lmax, 0) + 255) / 256, p->mmax + 2);
  tab_coef_k<<<cg, 256, 0, s>>>((const float2*)d_alm, p->lmax, p->mmax, a.M, p->leg.ahat, p->leg.pole_norm, t.ao,
                                (float2*)p->G);
  tab_synth_k<<<(t.nis + 3) / 4, 128, 0, s>>>(a, t.items_s, t.nis, t.ao, (float2*)p->G);
  NUSHT_CUDA(cudaGetLastError());
  return NUSHT_OK;
}

int legtab_adjoint(nusht_plan_t p, void* d_alm, cudaStream_t s, double wpos) {
  const LegTab& t = p->tab;
  const TabArgs a = args_of(p);
  const float2* Gt = (const float2*)p->Ghat;
  tab_adj_k<<<(t.nia + 3) / 4, 128, 0, s>>>(a, t.items_a, t.nia, Gt, (float4*)p->partial, t.n2);
  const dim3 rg((steps_of(p->lmax, 0) + 255) / 256, p->mmax + 1);
  tab_reduce_k<<<rg, 256, 0, s>>>(a, (a.ngrp + 3) / 4, (const float4*)p->partial, t.n2, p->leg.ahat, t.sc, t.w1, t.w2,
                                  p->leg.pole_norm, Gt, wpos, (float2*)d_alm);
  NUSHT_CUDA(cudaGetLastError());
  return NUSHT_OK;
}

}  // namespace nusht
