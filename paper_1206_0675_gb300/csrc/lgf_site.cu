// Site-local kernels of FA steepest-descent Landau gauge fixing:
//   * measure  : Delta(x), F and theta with a deterministic FP64 reduction
//                (arXiv:1206.0675 Sec. 2 and kernel k2 of Sec. 3.2),
//   * update   : U_mu(x) -> g(x) U_mu(x) g^dagger(x + mu^) (Sec. 2 eq. 2, kernel k6),
//   * layout conversion, SU(3) validation, the momentum filter table (k1).
// One thread per lattice site, or per link in the update of FP64 links; link
// arrays are structure-of-arrays so that a warp touches 32 consecutive sites of
// one matrix element per load.
#include <algorithm>
#include <cmath>

#include "lgf_fixed.cuh"
#include "lgf_internal.h"

namespace lgf {

// ---------------------------------------------------------------------------
// measure: Delta, F, theta
// ---------------------------------------------------------------------------

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Sum of a warp's FP64 values on the integer pipe: an FP64 addition holds its
// scheduler's FP64 pipe for 64 cycles, and five of them per value and warp were
// half of what the measurement of FP32 links spent.  The significands, aligned
// to the largest exponent of the warp with five bits below it, add exactly; what
// an alignment drops is below 2^-58 of the largest value, 32 of them below the
// 2^-53 of one FP64 rounding.  warp_align and warp_value frame the additions:
// q 2^(e - 1080) is the sum.
__device__ __forceinline__ int64_t warp_align(double v, uint32_t& e) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v), field = (hi >> 20) & 0x7ffu;
  const uint32_t ex = max(field, 1u);
  e = __reduce_max_sync(0xffffffffu, ex);
  const uint64_t m = ((uint64_t)((hi & 0xfffffu) | (field ? 0x100000u : 0u)) << 32) | lo;
  const int64_t q = (int64_t)((m << 5) >> min(e - ex, 63u));
  return (int32_t)hi < 0 ? -q : q;
}
__device__ __forceinline__ double warp_value(int64_t q, uint32_t e) {
  const double d = (double)q;
  const int hi = __double2hiint(d), ex = ((hi >> 20) & 0x7ff) + (int)e - 1080;
  if (q == 0) return 0.0;
  if (ex < 1 || ex > 2046) return d * 0x1p-57 * __hiloint2double((int)(e << 20), 0);
  return __hiloint2double(hi + (((int)e - 1080) << 20), __double2loint(d));
}

// Block reduction of two sums (fixed order) and a maximum of values >= 0 (FP32:
// the link defect is compared with bounds far above FP32 resolution; a NaN
// counts as 0), and of the warps' counts k; result valid in thread 0.  At most
// 16 warps.
__device__ __forceinline__ void block_reduce3(double& a, double& b, float& m, uint32_t& k) {
  __shared__ double sums[2][16];
  __shared__ uint32_t sm[16], sk[16];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  uint32_t ea, eb;
  int64_t qa = warp_align(a, ea), qb = warp_align(b, eb);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    qa += __shfl_xor_sync(0xffffffffu, qa, o);
    qb += __shfl_xor_sync(0xffffffffu, qb, o);
  }
  if (max(ea, eb) == 2047u) {  // infinities and NaN
    a = warp_sum(a);
    b = __shfl_sync(0xffffffffu, warp_sum(b), 0);
    if (lane < 2) sums[lane][warp] = lane == 0 ? a : b;
  } else {
    const double v = warp_value(lane == 0 ? qa : qb, lane == 0 ? ea : eb);
    if (lane < 2) sums[lane][warp] = v;
  }
  const uint32_t mw = __reduce_max_sync(0xffffffffu, m > 0.f ? __float_as_uint(m) : 0u);
  if (lane == 0) {
    sm[warp] = mw;
    sk[warp] = k;
  }
  __syncthreads();
  if (warp == 0) {
    const int w = lane & 15;
    double v = w < nw ? sums[lane >> 4][w] : 0.0;
    m = __uint_as_float(__reduce_max_sync(0xffffffffu, w < nw ? sm[w] : 0u));
    k = __reduce_add_sync(0xffffffffu, lane < nw ? sk[lane] : 0u);
    if (nw > 8) v += __shfl_xor_sync(0xffffffffu, v, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    a = v;
    b = __shfl_sync(0xffffffffu, v, 16);
  }
  __syncthreads();
}

// Unitarity defect of a link from its rows 1-2 (row 3 is always rebuilt as
// (a x b)^* or stored from that rebuild): the largest of | |a|^2 - 1 |,
// | |b|^2 - 1 | and the components of <a, b>, in the link precision.
template <typename R> __device__ __forceinline__ float rows_defect(const C2<R> a[3], const C2<R> b[3]) {
  const R na = cnorm2<R>(a[0]) + cnorm2<R>(a[1]) + cnorm2<R>(a[2]);
  const R nb = cnorm2<R>(b[0]) + cnorm2<R>(b[1]) + cnorm2<R>(b[2]);
  C2<R> ip = cconjmul<R>(a[0], b[0]);
  ip = cadd<R>(ip, cconjmul<R>(a[1], b[1]));
  ip = cadd<R>(ip, cconjmul<R>(a[2], b[2]));
  // the four deviations, each taken to FP32 before the maximum
  return fmaxf(fmaxf(fabsf((float)(na - (R)1)), fabsf((float)(nb - (R)1))),
               fmaxf(fabsf((float)ip.x), fabsf((float)ip.y)));
}

// The links whose defect a measurement samples: every sixteenth group of 32
// sites (group w with w % 16 == 0) takes direction (w / 16) % 4 of its 32
// sites, i.e. one link in 64, spread over all directions (the drift the
// guard watches is slow and lattice-wide).  The choice is uniform within a
// warp, so the other warps skip the work entirely.
__device__ __forceinline__ int defect_sample_mu(int64_t s) {
  const unsigned w = (unsigned)(s >> 5);
  return (w & 15u) == 0 ? (int)((w >> 4) & 3u) : -1;
}

// Reduction of the per-thread F and theta sums and the sampled link defect
// and, in the last CTA to finish, the controller update: F, theta and the
// defect, the iteration count, the history and its flags, the status word,
// the batch retirement flag or the graph's WHILE condition; flip_ubuf != 0
// also flips st->ubuf (after every CTA has read it); fp64 != 0 marks the
// measurement as one of FP64 links in the trace flags.
// fsum and tsum are the sums over the sites a thread collected, in FP64; every
// sum above a site (thread, warp, CTA, grid) is FP64 in a fixed order.  near_id:
// the warp's links are near the identity (FP64 links, the same in every lane);
// st->near_id is set where more than half of the warps' are.
__device__ __forceinline__ void measure_tail(const Geom& g, double fsum, double tsum, float dmax,
                                             double* __restrict__ partials, DevState* __restrict__ st, int count_iter,
                                             unsigned long long cond, int use_cond, bool batch, int flip_ubuf,
                                             int fp64, unsigned long long cond_undo, bool near_id) {
  double fb = fsum, tb = tsum;
  float db = dmax;
  uint32_t kb = near_id ? 1u : 0u;
  block_reduce3(fb, tb, db, kb);
  __shared__ uint32_t near_warps;
  __shared__ int is_last;
  if (threadIdx.x == 0) {
    partials[MEASURE_PARTIALS * blockIdx.x] = fb;
    partials[MEASURE_PARTIALS * blockIdx.x + 1] = tb;
    partials[MEASURE_PARTIALS * blockIdx.x + 2] = (double)db;
    __threadfence();
    const unsigned long long t = atomicAdd(&st->ticket, 1ull | ((unsigned long long)kb << 32));
    is_last = ((uint32_t)t == gridDim.x - 1);
    near_warps = (uint32_t)(t >> 32) + kb;
  }
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  // Final sum over the per-CTA partials in a fixed order (independent of
  // which CTA finished last), so the result is bit-reproducible.
  double f = 0.0, t = 0.0;
  float d = 0.f;
#pragma unroll 8
  for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) {
    f += __ldcg(&partials[MEASURE_PARTIALS * i]);
    t += __ldcg(&partials[MEASURE_PARTIALS * i + 1]);
    d = fmaxf(d, (float)__ldcg(&partials[MEASURE_PARTIALS * i + 2]));
  }
  block_reduce3(f, t, d, kb);
  if (threadIdx.x == 0) {
    const double Vd = (double)g.V;
    const double F = f / (12.0 * Vd);
    const double th = 4.0 * t / (3.0 * Vd);
    int it = st->iter;
    int revert = 0;
    int flags = fp64 ? TRACE_FP64 : 0;
    if (count_iter > 0) {
      it += count_iter;  // one FA step, or count_iter overrelaxation sweeps
      st->iter = it;
      st->F_prev = st->F;
      st->theta_prev = st->theta;
      // a learned step that lowered F is undone and redone with the plain filter
      if (st->use_m && F < st->F) {
        revert = 1;
        st->n_fallback += 1;
      }
      st->revert = revert;
      if (st->use_m) flags |= TRACE_LEARNED;
      if (st->redo) flags |= TRACE_REDO;
      if (st->repaired) flags |= TRACE_REPAIRED;
      st->redo = 0;
      st->repaired = 0;
    } else if (count_iter < 0) {
      it -= 1;
      st->iter = it;
    }
    st->snaps += count_iter;  // a rejected step's snapshot is replaced by its redo
    st->F = F;
    st->theta = th;
    st->defect = d;
    // The re-measurement after an undo repeats an entry already written; a
    // measurement without an update (after a precision switch or a repair)
    // refreshes F, theta and the defect of the current entry but keeps the
    // flags of the update that produced it.
    if (it < st->hist_cap && count_iter >= 0) {
      st->F_hist[it] = F;
      st->theta_hist[it] = th;
      if (st->flag_hist && count_iter > 0) st->flag_hist[it] = flags;
      if (st->defect_hist) st->defect_hist[it] = d;
    }
    const bool finite = isfinite(F) && isfinite(th);
    const bool sound = !(st->defect_bound > 0.0 && d > st->defect_bound);
    if (!finite) st->status = ST_NONFINITE;
    else if (!sound) st->status = ST_DEFECT;
    if (flip_ubuf) st->ubuf ^= 1;
    st->ticket = 0ull;
    st->near_id = 2u * near_warps > gridDim.x * (blockDim.x >> 5) ? 1 : 0;
    if (batch) st->done = !(finite && th >= st->tol && it < st->max_iter);
    if (use_cond) {
      cudaGraphConditionalHandle h = (cudaGraphConditionalHandle)cond;
      cudaGraphSetConditional(h, (finite && sound && ((th >= st->tol && it < st->max_iter) || revert)) ? 1u : 0u);
      if (cond_undo != 0 && count_iter > 0)
        cudaGraphSetConditional((cudaGraphConditionalHandle)cond_undo, revert ? 1u : 0u);
    }
  }
}

// ||Delta_A||_F^2 of the packed components, as an explicit FMA chain (the
// same rounding in every kernel that forms it).
template <typename R>
__device__ __forceinline__ R delta_norm2(R a0, R a1, R a2, C2<R> d01, C2<R> d02, C2<R> d12) {
  R off = d01.x * d01.x;
  off = fma(d01.y, d01.y, off);
  off = fma(d02.x, d02.x, off);
  off = fma(d02.y, d02.y, off);
  off = fma(d12.x, d12.x, off);
  off = fma(d12.y, d12.y, off);
  R dia = a0 * a0;
  dia = fma(a1, a1, dia);
  dia = fma(a2, a2, dia);
  return fma((R)2, off, dia);
}

// What one link M adds to a site's sums W = sum_mu [U_mu(x - mu^) - U_mu(x)]:
// Im M_ii and M_ij - conj(M_ji), the entries that enter the traceless
// anti-Hermitian part, and its trace.
template <typename R> struct LinkTerms {
  R tr, y0, y1, y2;
  C2<R> a01, a02, a12;
};
template <typename R> __device__ __forceinline__ LinkTerms<R> link_terms(const M3<R>& m) {
  LinkTerms<R> t;
  t.tr = m.e[0][0].x + m.e[1][1].x + m.e[2][2].x;
  t.y0 = m.e[0][0].y;
  t.y1 = m.e[1][1].y;
  t.y2 = m.e[2][2].y;
  t.a01 = csub<R>(m.e[0][1], cconj<R>(m.e[1][0]));
  t.a02 = csub<R>(m.e[0][2], cconj<R>(m.e[2][0]));
  t.a12 = csub<R>(m.e[1][2], cconj<R>(m.e[2][1]));
  return t;
}

// A site's sums: F's trace sum (FP32 links: as a pair f + fl, exact to 2^-46
// for the four traces it adds) and W in the link precision.
template <typename R> struct SiteSums {
  R f, fl;
  R im0, im1, im2;
  C2<R> w01, w02, w12;
};
__device__ __forceinline__ double sum_f(const SiteSums<double>& o) { return o.f; }
__device__ __forceinline__ double sum_f(const SiteSums<float>& o) { return f32_to_f64(o.f) + f32_to_f64(o.fl); }
__device__ __forceinline__ void add_f(SiteSums<double>& o, double x) { o.f += x; }
__device__ __forceinline__ void add_f(SiteSums<float>& o, float x) {
  const float s = __fadd_rn(o.f, x), t = __fsub_rn(s, o.f);
  o.fl += __fadd_rn(__fsub_rn(o.f, __fsub_rn(s, t)), __fsub_rn(x, t));
  o.f = s;
}
template <typename R> __device__ __forceinline__ SiteSums<R> site_sums_zero() {
  SiteSums<R> o;
  o.f = o.fl = 0;
  o.im0 = o.im1 = o.im2 = 0;
  o.w01 = o.w02 = o.w12 = mkc<R>(0, 0);
  return o;
}
// A site's own link of a direction, and the link of it that ends in the site.
template <typename R> __device__ __forceinline__ void add_own(SiteSums<R>& o, const LinkTerms<R>& t) {
  add_f(o, t.tr);
  o.im0 -= t.y0; o.im1 -= t.y1; o.im2 -= t.y2;
  o.w01 = csub<R>(o.w01, t.a01);
  o.w02 = csub<R>(o.w02, t.a02);
  o.w12 = csub<R>(o.w12, t.a12);
}
template <typename R> __device__ __forceinline__ void add_back(SiteSums<R>& o, const LinkTerms<R>& t) {
  o.im0 += t.y0; o.im1 += t.y1; o.im2 += t.y2;
  o.w01 = cadd<R>(o.w01, t.a01);
  o.w02 = cadd<R>(o.w02, t.a02);
  o.w12 = cadd<R>(o.w12, t.a12);
}

// Place of a thread of a measuring kernel: its site and the directions mu0 <=
// mu < mu1 of it.  SPLIT: eight sites to a warp (a whole 128-byte line of each
// FP64 entry), a lane per direction; lanes 0 to 7 go on with the sites' sums.
template <bool SPLIT> struct MeasurePlace {
  int64_t s;
  int mu0, mu1;
  __device__ __forceinline__ MeasurePlace() {
    if (SPLIT) {
      s = ((int64_t)blockIdx.x * (MEASURE_SPLIT_THREADS / 32) + (threadIdx.x >> 5)) * 8 + (threadIdx.x & 7);
      mu0 = (threadIdx.x >> 3) & 3;
      mu1 = mu0 + 1;
    } else {
      s = (int64_t)blockIdx.x * MEASURE_THREADS + threadIdx.x;
      mu0 = 0;
      mu1 = 4;
    }
  }
  static __device__ __forceinline__ bool collects() { return !SPLIT || (threadIdx.x & 24) == 0; }
  // the sum over the directions, in every lane of a site; all lanes of a warp call it
  template <typename T> static __device__ __forceinline__ void join(T& v) {
    if (SPLIT) {
      v += __shfl_xor_sync(0xffffffffu, v, 8);
      v += __shfl_xor_sync(0xffffffffu, v, 16);
    }
  }
  static __device__ __forceinline__ void join_or(uint32_t& v) {
    if (SPLIT) {
      v |= __shfl_xor_sync(0xffffffffu, v, 8);
      v |= __shfl_xor_sync(0xffffffffu, v, 16);
    }
  }
  static __device__ __forceinline__ void join(SiteSums<float>& o) {
    if (SPLIT) {
#pragma unroll
      for (int h = 8; h <= 16; h *= 2) {
        const float f = __shfl_xor_sync(0xffffffffu, o.f, h), fl = __shfl_xor_sync(0xffffffffu, o.fl, h);
        add_f(o, f);
        o.fl += fl;
      }
      join(o.im0); join(o.im1); join(o.im2);
      join(o.w01.x); join(o.w01.y); join(o.w02.x); join(o.w02.y); join(o.w12.x); join(o.w12.y);
    }
  }
  static __device__ __forceinline__ void join(SiteSums<double>& o) {
    if (SPLIT) {
      join(o.f); join(o.im0); join(o.im1); join(o.im2);
      join(o.w01.x); join(o.w01.y); join(o.w02.x); join(o.w02.y); join(o.w12.x); join(o.w12.y);
    }
  }
};

// Delta of a site, stored, and its part of theta.
template <typename R>
__device__ __forceinline__ double store_delta(const SiteSums<R>& o, C2<R>* __restrict__ delta, int64_t V, int64_t s) {
  const R tr = (o.im0 + o.im1 + o.im2) * (R)(1.0 / 3.0);
  const R a0 = o.im0 - tr, a1 = o.im1 - tr, a2 = o.im2 - tr;
  const C2<R> d01 = cscale<R>(o.w01, (R)0.5), d02 = cscale<R>(o.w02, (R)0.5), d12 = cscale<R>(o.w12, (R)0.5);
  delta[s] = mkc<R>(a0, a1);
  delta[V + s] = d01;
  delta[2 * V + s] = d02;
  delta[3 * V + s] = d12;
  // ||Delta_A||_F^2
  const R n = delta_norm2<R>(a0, a1, a2, d01, d02, d12);
  if constexpr (sizeof(R) == sizeof(float)) return f32_to_f64(n);
  else return n;
}

// A site's sums over its directions mu0 <= mu < mu0 + NMU in FP64: links near the
// identity and entries outside the fixed-point range.
template <int ROWS, int NMU>
__device__ __noinline__ void site_sums_fp64(const Geom& g, const MatField<double, ROWS>& U, int64_t s, int mu0,
                                            SiteSums<double>& o) {
  int c[4];
  site_coords(g, s, c);
  o = site_sums_zero<double>();
#pragma unroll
  for (int k = 0; k < NMU; ++k) {
    const int mu = mu0 + k;
    int64_t sf, sb;
    site_nbrs_sel(g, s, c, mu, sf, sb);
    M3<double> u, b;
    U.load_ro(mu, s, u);
    U.load_ro(mu, sb, b);
    add_own<double>(o, link_terms<double>(u));
    add_back<double>(o, link_terms<double>(b));
  }
}

// FP64 links: a site's sums over the two links of its directions mu0 <= mu < mu1 in 64-bit fixed point (unit 2^-58) on the integer
// pipe: exact but for what lies below 2^-58 in an entry, against one FP64
// rounding per addition (2^-54 for sums of order one).  12-real links rebuild
// row 3 in fixed point as well.
// t[0]: trace; t[1..3]: Im W_ii; t[4..9]: W_01, W_02, W_12; bad: an entry outside
// the range.  Returns false, for the whole warp, where the site's own link of
// direction mu0 is near the identity in any lane (FX_NEAR_HI).
constexpr int FX_TERMS = 10;
template <int ROWS>
__device__ __forceinline__ bool site_terms_fx(const Geom& g, const MatField<double, ROWS>& U, int64_t s,
                                              const int c[4], int mu0, int mu1, int64_t t[FX_TERMS], uint32_t& bad) {
  uint32_t m = 0, big = 0;
#pragma unroll 1
  for (int k = 2 * mu0; k < 2 * mu1; ++k) {
    const int mu = k >> 1;
    const bool own = (k & 1) == 0;
    int64_t sf, sb;
    site_nbrs_sel(g, s, c, mu, sf, sb);
    double2 e[ROWS][3];
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        e[r][j] = __ldg(&U.p[U.off(mu, r, j, own ? s : sb)]);
        m = fx_max(m, e[r][j]);
      }
    if (k == 2 * mu0 &&
        __any_sync(0xffffffffu, fx_max(fx_max(fx_max(0u, e[0][1]), e[0][2]), e[1][2]) < FX_NEAR_HI))
      return false;
    int64_t x[FX_TERMS];
    x[0] = 0;
    x[1] = fx58_from(e[0][0].y);
    x[2] = fx58_from(e[1][1].y);
    if (ROWS == 3) {
      if (own) x[0] = fx58_from(e[0][0].x) + fx58_from(e[1][1].x) + fx58_from(e[ROWS - 1][2].x);
      x[3] = fx58_from(e[ROWS - 1][2].y);
      x[4] = fx58_from(e[0][1].x) - fx58_from(e[1][0].x);
      x[5] = fx58_from(e[0][1].y) + fx58_from(e[1][0].y);
      x[6] = fx58_from(e[0][2].x) - fx58_from(e[ROWS - 1][0].x);
      x[7] = fx58_from(e[0][2].y) + fx58_from(e[ROWS - 1][0].y);
      x[8] = fx58_from(e[1][2].x) - fx58_from(e[ROWS - 1][1].x);
      x[9] = fx58_from(e[1][2].y) + fx58_from(e[ROWS - 1][1].y);
    } else {
      int64_t q[2][3][2], z[3][2];
      FxC w[2][3];
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          q[r][j][0] = fx58_from(e[r][j].x);
          q[r][j][1] = fx58_from(e[r][j].y);
          w[r][j] = FxC{fx_operand58(q[r][j][0]), fx_operand58(q[r][j][1])};
        }
      fx_third_row(w[0], w[1], z, big);
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        z[j][0] >>= 2;
        z[j][1] >>= 2;
      }
      if (own) x[0] = q[0][0][0] + q[1][1][0] + z[2][0];
      x[3] = z[2][1];
      x[4] = q[0][1][0] - q[1][0][0];
      x[5] = q[0][1][1] + q[1][0][1];
      x[6] = q[0][2][0] - z[0][0];
      x[7] = q[0][2][1] + z[0][1];
      x[8] = q[1][2][0] - z[1][0];
      x[9] = q[1][2][1] + z[1][1];
    }
    t[0] += x[0];
    if (own) {
#pragma unroll
      for (int i = 1; i < FX_TERMS; ++i) t[i] -= x[i];
    } else {
#pragma unroll
      for (int i = 1; i < FX_TERMS; ++i) t[i] += x[i];
    }
  }
  bad = fx_bad(m, big);
  return true;
}

// A site's sums from its directions' terms t; entries outside the fixed-point
// range take the FP64 path.
template <int ROWS>
__device__ __forceinline__ void site_sums_fx(const Geom& g, const MatField<double, ROWS>& U, int64_t s,
                                             const int64_t t[FX_TERMS], bool bad, SiteSums<double>& o) {
  if (bad) {
    site_sums_fp64<ROWS, 4>(g, U, s, 0, o);
    return;
  }
  o.f = fx_to_double_fp<58>(t[0]);
  o.im0 = fx_to_double_fp<58>(t[1]);
  o.im1 = fx_to_double_fp<58>(t[2]);
  o.im2 = fx_to_double_fp<58>(t[3]);
  o.w01 = make_double2(fx_to_double_fp<58>(t[4]), fx_to_double_fp<58>(t[5]));
  o.w02 = make_double2(fx_to_double_fp<58>(t[6]), fx_to_double_fp<58>(t[7]));
  o.w12 = make_double2(fx_to_double_fp<58>(t[8]), fx_to_double_fp<58>(t[9]));
}

// FP64 links are bound by the ALU pipe (66 % busy in ncu) beside HBM (40 %) and
// the FP64 pipe (41 %: the sites' conversions and norms).
// 32^4: 18-real 194 us (FP64 sums on the FP64 pipe: 355 us), 12-real 272 us
// (665 us); fields near the identity, whose warps take FP64 sums, 344 and 656 us.
template <typename R, int ROWS, bool SPLIT>
__global__ void __launch_bounds__(SPLIT ? MEASURE_SPLIT_THREADS : MEASURE_THREADS,
                                  SPLIT ? 1 : sizeof(R) == sizeof(float) ? 5 : ROWS == 3 ? 3 : 2)
measure_kernel(Geom g, MatField<R, ROWS> U, const C2<R>* __restrict__ links_alt, C2<R>* __restrict__ delta,
               double* __restrict__ partials, DevState* __restrict__ st, int count_iter, unsigned long long cond,
               int use_cond, int only_if_revert, Batch B, unsigned long long cond_undo) {
  if (batch_skip(B)) return;
  const bool batch = B.st != nullptr;
  if (batch) {
    const int cfg = blockIdx.z;
    st = B.st + cfg;
    U.p += cfg * B.s_links;
    delta += cfg * B.s_delta;
    partials += cfg * B.s_part;
  }
  if (only_if_revert && !st->revert) return;
  if (links_alt != nullptr && st->ubuf) U.p = const_cast<C2<R>*>(links_alt);  // ping-pong links of a fused lane
  const MeasurePlace<SPLIT> p;
  const bool in = p.s < g.V;
  // Re Tr of one link in the link precision; every sum above one link (the
  // site's F and theta terms, warp, CTA and grid sums) in FP64
  double fsum = 0, tsum = 0;
  float dmax = 0.f;
  int c[4];
  const int64_t sc = in ? p.s : g.V - 1;  // lanes past the end follow their warp
  site_coords(g, sc, c);
  bool near_id = false;
  // W = sum_mu [U_mu(x - mu^) - U_mu(x)]; only the entries that enter its
  // traceless anti-Hermitian part are accumulated.
  SiteSums<R> o = site_sums_zero<R>();
  if constexpr (sizeof(R) == sizeof(double)) {
    int64_t t[FX_TERMS] = {};
    uint32_t bad = 0;
    near_id = !site_terms_fx<ROWS>(g, U, sc, c, p.mu0, p.mu1, t, bad);
    if (!near_id) {
#pragma unroll
      for (int i = 0; i < FX_TERMS; ++i) p.join(t[i]);
      p.join_or(bad);
      if (in && p.collects()) site_sums_fx<ROWS>(g, U, p.s, t, bad != 0, o);
    } else {
      site_sums_fp64<ROWS, SPLIT ? 1 : 4>(g, U, sc, p.mu0, o);
      p.join(o);
    }
  } else {
    if (in) {
#pragma unroll
      for (int k = 0; k < (SPLIT ? 1 : 4); ++k) {
        const int mu = p.mu0 + k;
        int64_t sf, sb;
        site_nbrs_sel(g, p.s, c, mu, sf, sb);
        M3<R> u, b;
        U.load_ro(mu, p.s, u);
        add_own<R>(o, link_terms<R>(u));
        U.load_ro(mu, sb, b);
        add_back<R>(o, link_terms<R>(b));
      }
    }
    p.join(o);
  }
  if (in && p.collects()) {
    fsum = sum_f(o);
    tsum = store_delta<R>(o, delta, g.V, p.s);
    const int dmu = defect_sample_mu(p.s);
    if (dmu >= 0) {
      C2<R> rows[2][3];
      U.load_rows01_ro(dmu, p.s, rows);
      dmax = rows_defect<R>(rows[0], rows[1]);
    }
  }
  measure_tail(g, fsum, tsum, dmax, partials, st, count_iter, cond, use_cond, batch, 0, sizeof(R) == 8, cond_undo,
               near_id);
}

template <typename R, int ROWS>
cudaError_t launch_measure(const Geom& g, const C2<R>* links, C2<R>* delta, double* partials, DevState* st,
                           int count_iter, unsigned long long cond_handle, int use_cond, cudaStream_t s,
                           int only_if_revert, const Batch& B, const C2<R>* links_alt,
                           unsigned long long cond_undo) {
  const MatField<R, ROWS> U{const_cast<C2<R>*>(links), g.V};
  const dim3 grid((unsigned)measure_blocks(g.V), 1, (unsigned)B.n);
  if (measure_split(g.V))
    measure_kernel<R, ROWS, true><<<grid, MEASURE_SPLIT_THREADS, 0, s>>>(
        g, U, links_alt, delta, partials, st, count_iter, cond_handle, use_cond, only_if_revert, B, cond_undo);
  else
    measure_kernel<R, ROWS, false><<<grid, MEASURE_THREADS, 0, s>>>(
        g, U, links_alt, delta, partials, st, count_iter, cond_handle, use_cond, only_if_revert, B, cond_undo);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// fused update + measure (ping-pong links, backward neighbours recomputed)
// ---------------------------------------------------------------------------

// o = g u h^dagger: rows 0, 1 by products, row 2 = (row0 x row1)^* -- the
// same arithmetic as update_kernel, so that a recomputed neighbour link is
// bit-identical to the one its own thread stores.
template <typename R>
__device__ __forceinline__ void gauge_product(const M3<R>& gl, const M3<R>& u, const M3<R>& h, M3<R>& o) {
  C2<R> T[2][3];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      C2<R> acc = cmul_fx<R>(gl.e[i][0], u.e[0][j]);
      acc = cfma<R>(gl.e[i][1], u.e[1][j], acc);
      T[i][j] = cfma<R>(gl.e[i][2], u.e[2][j], acc);
    }
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      C2<R> acc = cmulc_fx<R>(T[i][0], h.e[j][0]);
      acc = cfmac<R>(T[i][1], h.e[j][1], acc);
      o.e[i][j] = cfmac<R>(T[i][2], h.e[j][2], acc);
    }
  su3_third_row<R>(o.e[0], o.e[1], o.e[2]);
}

template <typename R, int LROWS, int GROWS, bool SPLIT>
__global__ void __launch_bounds__(SPLIT ? MEASURE_SPLIT_THREADS : MEASURE_THREADS, 3)
update_measure_kernel(Geom g, C2<R>* __restrict__ U0, C2<R>* __restrict__ U1, MatField<R, GROWS> Gf,
                      C2<R>* __restrict__ delta, double* __restrict__ partials, DevState* __restrict__ st,
                      unsigned long long cond, int use_cond, unsigned long long cond_undo) {
  const int cur = st->ubuf;
  const MatField<R, LROWS> Us{cur ? U1 : U0, g.V}, Ud{cur ? U0 : U1, g.V};
  const MeasurePlace<SPLIT> p;
  const bool in = p.s < g.V;
  double fsum = 0, tsum = 0;  // as in measure_kernel: FP64 above one link
  float dmax = 0.f;
  SiteSums<R> o = site_sums_zero<R>();
  const int dmu = defect_sample_mu(p.s);
  if (in) {
    int c[4];
    site_coords(g, p.s, c);
    M3<R> gx;
    Gf.load_ro(0, p.s, gx);
#pragma unroll 1
    for (int mu = p.mu0; mu < p.mu1; ++mu) {
      M3<R> u, h, w;
      Us.load_ro(mu, p.s, u);
      Gf.load_ro(0, site_fwd(g, p.s, c, mu), h);
      gauge_product<R>(gx, u, h, w);
      Ud.store(mu, p.s, w);
      add_own<R>(o, link_terms<R>(w));
      const int64_t sb = site_back(g, p.s, c, mu);
      M3<R> b, gb, wb;
      Us.load_ro(mu, sb, b);
      Gf.load_ro(0, sb, gb);
      gauge_product<R>(gb, b, gx, wb);
      add_back<R>(o, link_terms<R>(wb));
    }
    if (dmu >= p.mu0 && dmu < p.mu1) {
      // the sampled link as this thread stored it above (plain loads see the
      // thread's own stores; keeping the rows in registers instead spilled)
      C2<R> rows[2][3];
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int j = 0; j < 3; ++j) rows[r][j] = Ud.p[Ud.off(dmu, r, j, p.s)];
      dmax = rows_defect<R>(rows[0], rows[1]);
    }
  }
  p.join(o);
  if (in && p.collects()) {
    fsum = sum_f(o);
    tsum = store_delta<R>(o, delta, g.V, p.s);
  }
  measure_tail(g, fsum, tsum, dmax, partials, st, 1, cond, use_cond, false, 1, sizeof(R) == 8, cond_undo, false);
}

template <typename R, int LROWS, int GROWS>
cudaError_t launch_update_measure(const Geom& g, C2<R>* U0, C2<R>* U1, const C2<R>* gfield, C2<R>* delta,
                                  double* partials, DevState* st, unsigned long long cond, int use_cond,
                                  cudaStream_t s, unsigned long long cond_undo) {
  MatField<R, GROWS> Gf{const_cast<C2<R>*>(gfield), g.V};
  const unsigned nb = (unsigned)measure_blocks(g.V);
  if (measure_split(g.V))
    update_measure_kernel<R, LROWS, GROWS, true><<<nb, MEASURE_SPLIT_THREADS, 0, s>>>(g, U0, U1, Gf, delta, partials,
                                                                                      st, cond, use_cond, cond_undo);
  else
    update_measure_kernel<R, LROWS, GROWS, false><<<nb, MEASURE_THREADS, 0, s>>>(g, U0, U1, Gf, delta, partials, st,
                                                                                 cond, use_cond, cond_undo);
  return cudaGetLastError();
}

__global__ void batch_condition_kernel(const DevState* __restrict__ st, int n, unsigned long long cond) {
  __shared__ int any;
  if (threadIdx.x == 0) any = 0;
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += blockDim.x)
    if (!st[i].done) any = 1;
  __syncthreads();
  if (threadIdx.x == 0) cudaGraphSetConditional((cudaGraphConditionalHandle)cond, any ? 1u : 0u);
}

cudaError_t launch_batch_condition(const DevState* st, int n, unsigned long long cond, cudaStream_t s) {
  batch_condition_kernel<<<1, 256, 0, s>>>(st, n, cond);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// update: U_mu(x) <- g(x) U_mu(x) g^dagger(x + mu^)
// ---------------------------------------------------------------------------

constexpr int UPDATE_THREADS = 128;

template <typename R, int LROWS, int GROWS>
__global__ void __launch_bounds__(UPDATE_THREADS)
update_kernel(Geom g, MatField<R, LROWS> U, MatField<R, GROWS> Gf, Batch B) {
  if (batch_skip(B)) return;
  U.p += blockIdx.z * B.s_links;
  Gf.p += blockIdx.z * B.s_g;
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  int c[4];
  site_coords(g, s, c);
  C2<R> gx[2][3];
  Gf.load_rows01_ro(0, s, gx);  // rows 1-2 of g(x) are all the product needs
#pragma unroll 1
  for (int mu = 0; mu < 4; ++mu) {
    M3<R> u;
    U.load(mu, s, u);
    M3<R> h;
    int64_t sf, sb;
    site_nbrs_sel(g, s, c, mu, sf, sb);  // selects: no local-memory copy of c[] in the loop
    Gf.load_ro(0, sf, h);
    // T = g(x)[rows 0,1] * U
    C2<R> T[2][3];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        C2<R> acc = cmul_fx<R>(gx[i][0], u.e[0][j]);
        acc = cfma<R>(gx[i][1], u.e[1][j], acc);
        T[i][j] = cfma<R>(gx[i][2], u.e[2][j], acc);
      }
    // rows 0,1 of T h^dagger; row 2 = (row0 x row1)^* (the result is in SU(3))
    M3<R> o;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        C2<R> acc = cmulc_fx<R>(T[i][0], h.e[j][0]);
        acc = cfmac<R>(T[i][1], h.e[j][1], acc);
        o.e[i][j] = cfmac<R>(T[i][2], h.e[j][2], acc);
      }
    if (LROWS == 3) su3_third_row<R>(o.e[0], o.e[1], o.e[2]);
    U.store(mu, s, o);
  }
}

// The FP64 path of one link: near the identity, or outside the fixed-point range.
template <int LROWS>
__device__ __noinline__ void update_link_fp64(MatField<double, LROWS> U, MatField<double, 3> Gf, int mu, int64_t s,
                                              int64_t sf) {
  M3<double> gx, u, h, o;
  fxg_load(Gf.p, Gf.V, s, gx);
  U.load(mu, s, u);
  fxg_load(Gf.p, Gf.V, sf, h);
  gauge_product<double>(gx, u, h, o);
  U.store(mu, s, o);
}

// FP64 links: the two products and row 3 in fixed point on the integer pipe
// (lgf_fixed.cuh); g arrives as operands.
// Fields near the identity (DevState::near_id) and warps with such links
// (FX_WEAK_HI) take FP64 before any arithmetic; links that meet a g in FP64 or
// have entries outside the fixed-point range take it after.  Error of one update against 64 bits at 32^4, eps = 1: 20 steps
// end at 2.4e-15 (FP64 products: 2.6e-15).
// Bound by the integer pipe (1780 instructions a link, 504 of them IMAD.WIDE,
// which run at about 30 of their 64 lanes a clock when all operands vary).
// 32^4, us: 18-real 379, 12-real 338; with FP64 products 1176 and 1177 at 95 %
// of the FP64 pipe (fields near the identity: 1191 and 1182).
// One thread per link: a CTA takes 32 sites, one direction per warp, so that
// the operand loads of a link are all in flight before its arithmetic and g(x)
// comes from L1 for three of the four warps.  The test for links near the
// identity stands between the loads of the link and those of g: after both it
// held all 24 in registers (393 us), and the CTAs of an SM hide the wait.
template <int LROWS>
__global__ void __launch_bounds__(UPDATE_THREADS, 5)
update_fx_kernel(Geom g, MatField<double, LROWS> U, MatField<double, 3> Gf, const DevState* __restrict__ st,
                 Batch B) {
  if (batch_skip(B)) return;
  const bool near_id = near_identity(st, B);
  U.p += blockIdx.z * B.s_links;
  Gf.p += blockIdx.z * B.s_g;
  const int64_t s0 = (int64_t)blockIdx.x * 32 + (threadIdx.x & 31);
  const int64_t s = min(s0, g.V - 1);  // lanes past the end follow their warp
  const bool in = s0 < g.V;
  const int mu = threadIdx.x >> 5;
  int c[4];
  site_coords(g, s, c);
  int64_t sf, sb;
  site_nbrs_sel(g, s, c, mu, sf, sb);
  const int4* G = reinterpret_cast<const int4*>(Gf.p);
  double2 u[LROWS][3];
  int4 g4[2][3], h4[3][3];
#pragma unroll
  for (int i = 0; i < LROWS; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) u[i][j] = U.p[U.off(mu, i, j, s)];
  if (__any_sync(0xffffffffu,
                 near_id || fx_max(fx_max(fx_max(0u, u[0][1]), u[0][2]), u[1][2]) < FX_WEAK_HI)) {
    if (in) update_link_fp64<LROWS>(U, Gf, mu, s, sf);
    return;
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) g4[i][j] = __ldg(&G[Gf.off(0, i, j, s)]);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) h4[i][j] = __ldg(&G[Gf.off(0, i, j, sf)]);
  uint32_t m = 0, t = 0;
#pragma unroll
  for (int i = 0; i < LROWS; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) m = fx_max(m, u[i][j]);
  // T = g(x)[rows 0,1] U
  FxC T[2][3], ux[3][3];
#pragma unroll
  for (int i = 0; i < LROWS; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) ux[i][j] = fx_from(u[i][j]);
  if (LROWS == 2) {
    int64_t c3[3][2];
    fx_third_row(ux[0], ux[1], c3, t);
#pragma unroll
    for (int j = 0; j < 3; ++j) ux[2][j] = FxC{fx_operand(c3[j][0]), fx_operand(c3[j][1])};
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    FxC gx[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) gx[k] = fxg_unpack(g4[i][k]);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      FxAcc re = fx_zero(), im = fx_zero();
#pragma unroll
      for (int k = 0; k < 3; ++k) fx_cmac(re, im, gx[k], fx_neg(gx[k].y), ux[k][j]);
      T[i][j] = FxC{fx_operand(fx_sum60(re, t)), fx_operand(fx_sum60(im, t))};
    }
  }
  // rows 0,1 of T h^dagger
  int64_t n[2][3][2];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      FxAcc re = fx_zero(), im = fx_zero();
#pragma unroll
      for (int k = 0; k < 3; ++k) fx_cmacc(re, im, T[i][k], fx_neg(T[i][k].x), fxg_unpack(h4[j][k]));
      n[i][j][0] = fx_sum60(re, t);
      n[i][j][1] = fx_sum60(im, t);
    }
  // row 3 of 18-real links: (row 1 x row 2)^*
  int64_t n3[3][2];
  if (LROWS == 3) {
    FxC r[2][3];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) r[i][j] = FxC{fx_operand(n[i][j][0]), fx_operand(n[i][j][1])};
    fx_third_row(r[0], r[1], n3, t);
  }
  if (!in) return;
  if (fx_bad(m, t) || fxg_is_fp64(g4[0][0]) || fxg_is_fp64(h4[0][0])) {
    update_link_fp64<LROWS>(U, Gf, mu, s, sf);
    return;
  }
  double2 o[LROWS][3];
  fx_link_to_double<LROWS>(n, n3, o);
#pragma unroll
  for (int i = 0; i < LROWS; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) U.p[U.off(mu, i, j, s)] = o[i][j];
}

template <typename R, int LROWS, int GROWS>
cudaError_t launch_update(const Geom& g, C2<R>* links, const C2<R>* gfield, const DevState* st, cudaStream_t s,
                          const Batch& B) {
  MatField<R, LROWS> U{links, g.V};
  MatField<R, GROWS> Gf{const_cast<C2<R>*>(gfield), g.V};
  const int64_t nb = (g.V + UPDATE_THREADS - 1) / UPDATE_THREADS;
  const dim3 grid((unsigned)nb, 1, (unsigned)B.n);
  if constexpr (sizeof(R) == sizeof(double)) {
    static_assert(GROWS == 3, "FP64 lanes keep three rows of g");
    const dim3 fx_grid((unsigned)((g.V + 31) / 32), 1, (unsigned)B.n);
    update_fx_kernel<LROWS><<<fx_grid, UPDATE_THREADS, 0, s>>>(g, U, Gf, st, B);
  } else {
    update_kernel<R, LROWS, GROWS><<<grid, UPDATE_THREADS, 0, s>>>(g, U, Gf, B);
  }
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// undo of a rejected step: U_mu(x) <- g^dag(x) U_mu(x) g(x + mu^), G <- g^dag G
// ---------------------------------------------------------------------------

// g(s) of a lane as a matrix (lgf_fixed.cuh has the forms of FP64 lanes).
template <int GROWS>
__device__ __forceinline__ void load_g(const MatField<float, GROWS>& Gf, int64_t s, M3<float>& M) {
  Gf.load_ro(0, s, M);
}
__device__ __forceinline__ void load_g(const MatField<double, 3>& Gf, int64_t s, M3<double>& M) {
  fxg_load(Gf.p, Gf.V, s, M);
}

template <typename R, int LROWS, int GROWS>
__global__ void __launch_bounds__(UPDATE_THREADS)
revert_kernel(Geom g, MatField<R, LROWS> U, MatField<R, GROWS> Gf, MatField<R, 3> Gacc, const DevState* st,
              C2<R>* links_alt) {
  if (!st->revert) return;
  if (links_alt != nullptr && st->ubuf) U.p = links_alt;  // the current buffer of a fused lane
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  int c[4];
  site_coords(g, s, c);
  M3<R> gx;
  load_g(Gf, s, gx);
#pragma unroll 1
  for (int mu = 0; mu < 4; ++mu) {
    M3<R> u, h;
    U.load(mu, s, u);
    load_g(Gf, site_fwd(g, s, c, mu), h);
    // T = (g^dag U)[rows 0,1]: T_ij = sum_k conj(g_ki) U_kj
    C2<R> T[2][3];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        C2<R> acc = cconjmul<R>(gx.e[0][i], u.e[0][j]);
        acc = cadd<R>(acc, cconjmul<R>(gx.e[1][i], u.e[1][j]));
        T[i][j] = cadd<R>(acc, cconjmul<R>(gx.e[2][i], u.e[2][j]));
      }
    M3<R> o;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        C2<R> acc = cmul<R>(T[i][0], h.e[0][j]);
        acc = cfma<R>(T[i][1], h.e[1][j], acc);
        o.e[i][j] = cfma<R>(T[i][2], h.e[2][j], acc);
      }
    su3_third_row<R>(o.e[0], o.e[1], o.e[2]);
    U.store(mu, s, o);
  }
  if (Gacc.p != nullptr) {
    M3<R> G0, G1;
    Gacc.load(0, s, G0);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        C2<R> acc = cconjmul<R>(gx.e[0][i], G0.e[0][j]);
        acc = cadd<R>(acc, cconjmul<R>(gx.e[1][i], G0.e[1][j]));
        G1.e[i][j] = cadd<R>(acc, cconjmul<R>(gx.e[2][i], G0.e[2][j]));
      }
    Gacc.store(0, s, G1);
  }
}

template <typename R, int LROWS, int GROWS>
cudaError_t launch_revert(const Geom& g, C2<R>* links, const C2<R>* gfield, C2<R>* Gacc, const DevState* st,
                          cudaStream_t s, C2<R>* links_alt) {
  MatField<R, LROWS> U{links, g.V};
  MatField<R, GROWS> Gf{const_cast<C2<R>*>(gfield), g.V};
  MatField<R, 3> Ga{Gacc, g.V};
  const int64_t nb = (g.V + UPDATE_THREADS - 1) / UPDATE_THREADS;
  revert_kernel<R, LROWS, GROWS><<<(unsigned)nb, UPDATE_THREADS, 0, s>>>(g, U, Gf, Ga, st, links_alt);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// layout conversion
// ---------------------------------------------------------------------------

constexpr int CONV_THREADS = 256;

// The user's layout keeps the nine entries of a matrix together (144 bytes):
// CTAs copy CONV_MATS matrices between it and shared memory as one contiguous
// run, and a thread takes its matrix from there (nine 16-byte words apart: no
// bank conflicts).  Read by each thread from its own matrix, the layout costs 32
// sectors per 16-byte load of a warp.  lgf_set_links at 32^4 with the check below
// in fixed point: 1573 -> 717 us (FP64), 1400 -> 475 us (FP32); lgf_get_links
// 450 -> 205 us, 370 -> 171 us (floors 89 us a pass over the links).
constexpr int CONV_MATS = 128;

__device__ __forceinline__ void aos_tile_load(double2* tile, const double2* __restrict__ aos, int64_t i0, int n) {
  const double2* src = aos + i0 * 9;
  const int m = 9 * n;
  if (n == CONV_MATS) {
    double2 v[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) v[k] = __ldg(&src[threadIdx.x + k * CONV_MATS]);
#pragma unroll
    for (int k = 0; k < 9; ++k) tile[threadIdx.x + k * CONV_MATS] = v[k];
  } else {
    for (int k = threadIdx.x; k < m; k += CONV_MATS) tile[k] = __ldg(&src[k]);
  }
  __syncthreads();
}
__device__ __forceinline__ void aos_tile_store(const double2* tile, double2* __restrict__ aos, int64_t i0, int n) {
  __syncthreads();
  double2* dst = aos + i0 * 9;
  for (int k = threadIdx.x; k < 9 * n; k += CONV_MATS) dst[k] = tile[k];
}

// Links use nmat = 4 (mu) matrices per site, site fields nmat = 1.
template <typename R, int ROWS>
__global__ void __launch_bounds__(CONV_MATS)
from_aos_kernel(int64_t V, int nmat, const double2* __restrict__ aos, MatField<R, ROWS> F) {
  __shared__ double2 tile[9 * CONV_MATS];
  const int64_t i0 = (int64_t)blockIdx.x * CONV_MATS;
  const int n = (int)min((int64_t)CONV_MATS, V * nmat - i0);
  aos_tile_load(tile, aos, i0, n);
  if ((int)threadIdx.x >= n) return;
  const int64_t i = i0 + threadIdx.x;
  const int m = nmat == 1 ? 0 : (int)((i >= V) + (i >= 2 * V) + (i >= 3 * V));
  const int64_t s = i - (int64_t)m * V;
#pragma unroll
  for (int e = 0; e < 3 * ROWS; ++e) {
    const double2 v = tile[threadIdx.x * 9 + e];
    if constexpr (sizeof(R) == sizeof(float))
      F.p[F.off(m, e / 3, e % 3, s)] = mkc<R>(f64_to_f32(v.x), f64_to_f32(v.y));
    else
      F.p[F.off(m, e / 3, e % 3, s)] = v;
  }
}

template <typename R, int ROWS>
__global__ void __launch_bounds__(CONV_MATS)
to_aos_kernel(int64_t V, int nmat, MatField<R, ROWS> F, double2* __restrict__ aos) {
  __shared__ double2 tile[9 * CONV_MATS];
  const int64_t i0 = (int64_t)blockIdx.x * CONV_MATS;
  const int n = (int)min((int64_t)CONV_MATS, V * nmat - i0);
  if ((int)threadIdx.x < n) {
    const int64_t i = i0 + threadIdx.x;
    const int m = nmat == 1 ? 0 : (int)((i >= V) + (i >= 2 * V) + (i >= 3 * V));
    M3<R> M;
    F.load_ro(m, i - (int64_t)m * V, M);
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      const C2<R> v = M.e[e / 3][e % 3];
      if constexpr (sizeof(R) == sizeof(float))
        tile[threadIdx.x * 9 + e] = make_double2(f32_to_f64(v.x), f32_to_f64(v.y));
      else
        tile[threadIdx.x * 9 + e] = v;
    }
  }
  aos_tile_store(tile, aos, i0, n);
}

static unsigned conv_blocks(int64_t nmat) { return (unsigned)((nmat + CONV_MATS - 1) / CONV_MATS); }

__global__ void __launch_bounds__(CONV_MATS)
gauge_to_aos_kernel(int64_t V, const double2* __restrict__ gf, double2* __restrict__ aos) {
  __shared__ double2 tile[9 * CONV_MATS];
  const int64_t i0 = (int64_t)blockIdx.x * CONV_MATS;
  const int n = (int)min((int64_t)CONV_MATS, V - i0);
  if ((int)threadIdx.x < n) {
    M3<double> M;
    fxg_load(gf, V, i0 + threadIdx.x, M);
#pragma unroll
    for (int e = 0; e < 9; ++e) tile[threadIdx.x * 9 + e] = M.e[e / 3][e % 3];
  }
  aos_tile_store(tile, aos, i0, n);
}

cudaError_t launch_gauge_to_aos(const Geom& g, const double2* gfield, double* aos, cudaStream_t s) {
  gauge_to_aos_kernel<<<conv_blocks(g.V), CONV_MATS, 0, s>>>(g.V, gfield, reinterpret_cast<double2*>(aos));
  return cudaGetLastError();
}

template <typename R, int ROWS>
cudaError_t launch_links_from_aos(const Geom& g, const double* aos, C2<R>* links, cudaStream_t s) {
  MatField<R, ROWS> F{links, g.V};
  const int64_t n = 4 * g.V;
  from_aos_kernel<R, ROWS><<<conv_blocks(n), CONV_MATS, 0, s>>>(g.V, 4, reinterpret_cast<const double2*>(aos), F);
  return cudaGetLastError();
}

template <typename R, int ROWS>
cudaError_t launch_links_to_aos(const Geom& g, const C2<R>* links, double* aos, cudaStream_t s) {
  MatField<R, ROWS> F{const_cast<C2<R>*>(links), g.V};
  const int64_t n = 4 * g.V;
  to_aos_kernel<R, ROWS><<<conv_blocks(n), CONV_MATS, 0, s>>>(g.V, 4, F, reinterpret_cast<double2*>(aos));
  return cudaGetLastError();
}

template <typename R, int ROWS>
cudaError_t launch_sites_to_aos(const Geom& g, const C2<R>* field, double* aos, cudaStream_t s) {
  MatField<R, ROWS> F{const_cast<C2<R>*>(field), g.V};
  to_aos_kernel<R, ROWS><<<conv_blocks(g.V), CONV_MATS, 0, s>>>(g.V, 1, F, reinterpret_cast<double2*>(aos));
  return cudaGetLastError();
}

template <typename R, int ROWS>
cudaError_t launch_sites_from_aos(const Geom& g, const double* aos, C2<R>* field, cudaStream_t s) {
  MatField<R, ROWS> F{field, g.V};
  from_aos_kernel<R, ROWS><<<conv_blocks(g.V), CONV_MATS, 0, s>>>(g.V, 1, reinterpret_cast<const double2*>(aos), F);
  return cudaGetLastError();
}

template <typename R>
__global__ void delta_to_aos_kernel(int64_t V, const C2<R>* __restrict__ d, double2* __restrict__ aos) {
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= V) return;
  const C2<R> f0 = d[s], f1 = d[V + s], f2 = d[2 * V + s], f3 = d[3 * V + s];
  const double a0 = f0.x, a1 = f0.y, a2 = -(a0 + a1);
  double2* o = aos + s * 9;
  o[0] = make_double2(0.0, a0);
  o[1] = make_double2(f1.x, f1.y);
  o[2] = make_double2(f2.x, f2.y);
  o[3] = make_double2(-(double)f1.x, (double)f1.y);
  o[4] = make_double2(0.0, a1);
  o[5] = make_double2(f3.x, f3.y);
  o[6] = make_double2(-(double)f2.x, (double)f2.y);
  o[7] = make_double2(-(double)f3.x, (double)f3.y);
  o[8] = make_double2(0.0, a2);
}

template <typename R>
cudaError_t launch_delta_to_aos(const Geom& g, const C2<R>* delta, double* aos, cudaStream_t s) {
  delta_to_aos_kernel<R><<<(unsigned)((g.V + CONV_THREADS - 1) / CONV_THREADS), CONV_THREADS, 0, s>>>(
      g.V, delta, reinterpret_cast<double2*>(aos));
  return cudaGetLastError();
}

template <typename R, int ROWS>
__global__ void identity_kernel(int64_t V, MatField<R, ROWS> F) {
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= V) return;
#pragma unroll
  for (int r = 0; r < ROWS; ++r)
#pragma unroll
    for (int c = 0; c < 3; ++c) F.p[F.off(0, r, c, s)] = mkc<R>(r == c ? (R)1 : (R)0, (R)0);
}

template <typename R, int ROWS>
cudaError_t launch_set_identity(const Geom& g, C2<R>* field, cudaStream_t s) {
  MatField<R, ROWS> F{field, g.V};
  identity_kernel<R, ROWS><<<(unsigned)((g.V + CONV_THREADS - 1) / CONV_THREADS), CONV_THREADS, 0, s>>>(g.V, F);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// SU(3) validation of user links
// ---------------------------------------------------------------------------

__device__ __noinline__ double su3_defect_fp64(const double2* mat) {
  double2 m[3][3];
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int c = 0; c < 3; ++c) m[r][c] = mat[r * 3 + c];
  double d = 0.0;
  // U U^dag is Hermitian: its upper triangle holds every distinct entry
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int c = r; c < 3; ++c) {
      double2 acc = mkc<double>(0.0, 0.0);
#pragma unroll
      for (int k = 0; k < 3; ++k) acc = cfmac<double>(m[r][k], m[c][k], acc);
      if (r == c) acc.x -= 1.0;
      d = fmax(d, fmax(fabs(acc.x), fabs(acc.y)));
    }
  double2 cr[3];
  su3_third_row<double>(m[0], m[1], cr);  // conj(r0 x r1)
  // det = r2 . (r0 x r1) = sum_j r2_j conj(cr_j)
  double2 det = mkc<double>(0.0, 0.0);
#pragma unroll
  for (int j = 0; j < 3; ++j) det = cfmac<double>(m[2][j], cr[j], det);
  d = fmax(d, sqrt((det.x - 1.0) * (det.x - 1.0) + det.y * det.y));
  bool finite = true;
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int c = 0; c < 3; ++c) finite = finite && isfinite(m[r][c].x) && isfinite(m[r][c].y);
  return (!finite || !isfinite(d)) ? INFINITY : d;
}

// The largest deviation of a matrix in fixed point, in units of 2^-60: entries
// of U U^dag - 1 and the components of det U - 1.  A matrix whose deviations
// all stay below SU3_CLEAR passes any test of the input (1e-10), so only
// others, and entries outside the fixed-point range, are formed in FP64.
// 90 real products on the integer pipe against about 110 FP64 operations.
constexpr int64_t SU3_CLEAR = (int64_t)(5e-11 * 1152921504606846976.0);  // 5e-11
__device__ __forceinline__ int64_t su3_defect_fx(const double2* mat, bool& bad) {
  uint32_t m = 0, t = 0;
  FxC u[3][3];
#pragma unroll
  for (int e = 0; e < 9; ++e) {
    const double2 v = mat[e];
    m = fx_max(m, v);
    u[e / 3][e % 3] = fx_from(v);
  }
  const int64_t one = (int64_t)1 << 60;
  int64_t d = 0;
  auto fold = [&](int64_t x) { d = max(d, x < 0 ? -x : x); };
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    FxAcc nn = fx_zero();
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      fx_mac(nn, u[r][k].x, u[r][k].x);
      fx_mac(nn, u[r][k].y, u[r][k].y);
    }
    fold(fx_sum60(nn, t) - one);
#pragma unroll
    for (int c = r + 1; c < 3; ++c) {
      FxAcc re = fx_zero(), im = fx_zero();
#pragma unroll
      for (int k = 0; k < 3; ++k) fx_cmacc(re, im, u[r][k], fx_neg(u[r][k].x), u[c][k]);
      fold(fx_sum60(re, t));
      fold(fx_sum60(im, t));
    }
  }
  int64_t c3[3][2];
  fx_third_row(u[0], u[1], c3, t);
  FxAcc re = fx_zero(), im = fx_zero();
#pragma unroll
  for (int j = 0; j < 3; ++j)
    fx_cmacc(re, im, u[2][j], fx_neg(u[2][j].x), FxC{fx_operand(c3[j][0]), fx_operand(c3[j][1])});
  fold(fx_sum60(re, t) - one);
  fold(fx_sum60(im, t));
  bad = fx_bad(m, t) || d >= SU3_CLEAR;
  return d;
}

// Grid-stride over tiles of matrices; the maximum of a CTA goes to *out by one
// atomic (a few thousand in all, instead of one per warp on one address).
__global__ void __launch_bounds__(CONV_MATS) su3_defect_kernel(const double2* __restrict__ aos, int64_t nmat,
                                                               unsigned long long* out) {
  __shared__ double2 tile[9 * CONV_MATS];
  double d = 0.0;
  int64_t dx = 0;
  for (int64_t i0 = (int64_t)blockIdx.x * CONV_MATS; i0 < nmat; i0 += (int64_t)gridDim.x * CONV_MATS) {
    const int n = (int)min((int64_t)CONV_MATS, nmat - i0);
    __syncthreads();
    aos_tile_load(tile, aos, i0, n);
    if ((int)threadIdx.x < n) {
      bool bad;
      const int64_t x = su3_defect_fx(tile + threadIdx.x * 9, bad);
      if (bad) d = fmax(d, su3_defect_fp64(tile + threadIdx.x * 9));
      else dx = max(dx, x);
    }
  }
  d = fmax(d, fx_to_double_fp<60>(dx));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) d = fmax(d, __shfl_down_sync(0xffffffffu, d, o));
  __shared__ double wm[CONV_MATS / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = CONV_MATS / 32;
  if (lane == 0) wm[warp] = d;
  __syncthreads();
  if (warp == 0) {
    d = lane < nw ? wm[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) d = fmax(d, __shfl_down_sync(0xffffffffu, d, o));
    if (lane == 0) atomicMax(out, (unsigned long long)__double_as_longlong(d));
  }
}

cudaError_t launch_su3_defect(const double* aos, int64_t nmat, unsigned long long* out_bits, cudaStream_t s,
                              int reset) {
  if (reset) {
    cudaError_t e = cudaMemsetAsync(out_bits, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
  }
  const int64_t blocks = std::min<int64_t>(conv_blocks(nmat), 152 * 8);
  su3_defect_kernel<<<(unsigned)(blocks > 0 ? blocks : 1), CONV_MATS, 0, s>>>(
      reinterpret_cast<const double2*>(aos), nmat, out_bits);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// momentum filter table (kernel k1 of Sec. 3.2)
// ---------------------------------------------------------------------------

template <typename R>
__global__ void filter_table_kernel(Geom g, const double* __restrict__ sin2, int lmax, double alpha, double p2max,
                                    int plain_sd, R* __restrict__ K) {
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  int c[4];
  site_coords(g, s, c);
  const double p2 = sin2[3 * lmax + c[3]] + sin2[2 * lmax + c[2]] + sin2[lmax + c[1]] + sin2[c[0]];
  double k = 0.0;
  if (s != 0) k = plain_sd ? alpha / (double)g.V : alpha * p2max / (p2 * (double)g.V);
  K[s] = (R)k;
}

template <typename R>
cudaError_t launch_filter_table(const Geom& g, const double* sin2, int lmax, double alpha, double p2max, int plain_sd,
                                R* K, cudaStream_t s) {
  filter_table_kernel<R><<<(unsigned)((g.V + CONV_THREADS - 1) / CONV_THREADS), CONV_THREADS, 0, s>>>(
      g, sin2, lmax, alpha, p2max, plain_sd, K);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// controller state, precision conversion, FP64 projection of G
// ---------------------------------------------------------------------------

__global__ void set_state_kernel(DevState* st, double tol, int max_iter, int reset_iter, int hist_cap, double* Fh,
                                 double* Th, int* flh, double* dfh, double defect_bound, int flags0) {
  st->tol = tol;
  st->max_iter = max_iter;
  if (reset_iter) {
    st->iter = 0;
    st->theta_prev = 0.0;
    st->status = ST_OK;
    st->revert = 0;
    st->use_m = 0;
    st->n_fallback = 0;
    st->redo = 0;
    st->repaired = 0;
    st->snaps = 0;
  }
  st->hist_cap = hist_cap;
  st->F_hist = Fh;
  st->theta_hist = Th;
  st->flag_hist = flh;
  st->defect_hist = dfh;
  st->defect_bound = defect_bound;
  if (hist_cap > 0 && reset_iter) {
    Fh[0] = st->F;
    Th[0] = st->theta;
    if (flh) flh[0] = flags0;
    if (dfh) dfh[0] = st->defect;
  }
}

cudaError_t launch_set_state(DevState* st, double tol, int max_iter, int reset_iter, int hist_cap, double* F_hist,
                             double* theta_hist, cudaStream_t s, int* flag_hist, double* defect_hist,
                             double defect_bound, int flags0) {
  set_state_kernel<<<1, 1, 0, s>>>(st, tol, max_iter, reset_iter, hist_cap, F_hist, theta_hist, flag_hist,
                                   defect_hist, defect_bound, flags0);
  return cudaGetLastError();
}

// Gram-Schmidt on rows 1-2 of every link, row 3 = (a x b)^* when stored.
template <typename R, int ROWS>
__global__ void reunitarize_links_kernel(int64_t n, MatField<R, ROWS> U) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int m = (int)(i / U.V);
  const int64_t s = i - (int64_t)m * U.V;
  M3<R> M;
  U.load(m, s, M);
  C2<R>* a = M.e[0];
  C2<R>* b = M.e[1];
  const R ia = (R)1 / sqrt(cnorm2<R>(a[0]) + cnorm2<R>(a[1]) + cnorm2<R>(a[2]));
#pragma unroll
  for (int j = 0; j < 3; ++j) a[j] = cscale<R>(a[j], ia);
  C2<R> ip = cconjmul<R>(a[0], b[0]);
  ip = cadd<R>(ip, cconjmul<R>(a[1], b[1]));
  ip = cadd<R>(ip, cconjmul<R>(a[2], b[2]));
  const C2<R> nip = mkc<R>(-ip.x, -ip.y);
#pragma unroll
  for (int j = 0; j < 3; ++j) b[j] = cfma<R>(nip, a[j], b[j]);
  const R ib = (R)1 / sqrt(cnorm2<R>(b[0]) + cnorm2<R>(b[1]) + cnorm2<R>(b[2]));
#pragma unroll
  for (int j = 0; j < 3; ++j) b[j] = cscale<R>(b[j], ib);
  su3_third_row<R>(M.e[0], M.e[1], M.e[2]);
  U.store(m, s, M);
}

__global__ void mark_repaired_kernel(DevState* st) {
  st->repaired = 1;
  if (st->status == ST_DEFECT) st->status = ST_OK;
}

template <typename R, int ROWS>
cudaError_t launch_reunitarize_links(const Geom& g, C2<R>* links, DevState* st, cudaStream_t s) {
  MatField<R, ROWS> U{links, g.V};
  const int64_t n = 4 * g.V;
  reunitarize_links_kernel<R, ROWS><<<(unsigned)((n + CONV_THREADS - 1) / CONV_THREADS), CONV_THREADS, 0, s>>>(n, U);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  mark_repaired_kernel<<<1, 1, 0, s>>>(st);
  return cudaGetLastError();
}

__global__ void c2_f64_to_f32_kernel(const double2* __restrict__ in, float2* __restrict__ out, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = make_float2((float)in[i].x, (float)in[i].y);
}

__global__ void c2_f32_to_f64_kernel(const float2* __restrict__ in, double2* __restrict__ out, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = make_double2((double)in[i].x, (double)in[i].y);
}

cudaError_t launch_c2_f64_to_f32(const double2* in, float2* out, int64_t n, cudaStream_t s) {
  c2_f64_to_f32_kernel<<<(unsigned)((n + CONV_THREADS - 1) / CONV_THREADS), CONV_THREADS, 0, s>>>(in, out, n);
  return cudaGetLastError();
}

cudaError_t launch_c2_f32_to_f64(const float2* in, double2* out, int64_t n, cudaStream_t s) {
  c2_f32_to_f64_kernel<<<(unsigned)((n + CONV_THREADS - 1) / CONV_THREADS), CONV_THREADS, 0, s>>>(in, out, n);
  return cudaGetLastError();
}

// Gram-Schmidt projection of rows 1-2 to SU(3) in FP64, row 3 = (a x b)^*,
// as g of the FP64 lane and, where it tracks the transform, as its G.  links: the
// input links (user layout) that g is about to transform; near the identity it
// is kept in FP64.
__global__ void project_sites_kernel(int64_t V, const float2* __restrict__ in, const double2* __restrict__ links,
                                     double2* __restrict__ gf, double2* __restrict__ out) {
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= V) return;
  double2 a[3], b[3], c[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const float2 x = in[(0 * 3 + j) * V + s], y = in[(1 * 3 + j) * V + s];
    a[j] = make_double2(x.x, x.y);
    b[j] = make_double2(y.x, y.y);
  }
  const double ia = rsqrt(cnorm2<double>(a[0]) + cnorm2<double>(a[1]) + cnorm2<double>(a[2]));
#pragma unroll
  for (int j = 0; j < 3; ++j) a[j] = cscale<double>(a[j], ia);
  double2 ip = cconjmul<double>(a[0], b[0]);
  ip = cadd<double>(ip, cconjmul<double>(a[1], b[1]));
  ip = cadd<double>(ip, cconjmul<double>(a[2], b[2]));
  const double2 nip = make_double2(-ip.x, -ip.y);
#pragma unroll
  for (int j = 0; j < 3; ++j) b[j] = cfma<double>(nip, a[j], b[j]);
  const double ib = rsqrt(cnorm2<double>(b[0]) + cnorm2<double>(b[1]) + cnorm2<double>(b[2]));
#pragma unroll
  for (int j = 0; j < 3; ++j) b[j] = cscale<double>(b[j], ib);
  su3_third_row<double>(a, b, c);
  bool near_id = false;
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    const double2* u = links + (mu * V + s) * 9;
    near_id = near_id || fx_max(fx_max(fx_max(0u, __ldg(u + 1)), __ldg(u + 2)), __ldg(u + 5)) < FX_NEAR_HI;
  }
  if (near_id) fxg_store_fp64(gf, V, s, a, b, c);
  else fxg_store(gf, V, s, a, b, c);
  if (out == nullptr) return;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    out[(0 * 3 + j) * V + s] = a[j];
    out[(1 * 3 + j) * V + s] = b[j];
    out[(2 * 3 + j) * V + s] = c[j];
  }
}

cudaError_t launch_project_sites_f32_to_f64(const Geom& g, const float2* G32, const double* links, double2* gfield,
                                            double2* G64, cudaStream_t s) {
  project_sites_kernel<<<(unsigned)((g.V + CONV_THREADS - 1) / CONV_THREADS), CONV_THREADS, 0, s>>>(
      g.V, G32, reinterpret_cast<const double2*>(links), gfield, G64);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// explicit instantiations
// ---------------------------------------------------------------------------

#define LGF_INST_R_ROWS(R, ROWS)                                                                                     \
  template cudaError_t launch_measure<R, ROWS>(const Geom&, const C2<R>*, C2<R>*, double*, DevState*, int,           \
                                               unsigned long long, int, cudaStream_t, int, const Batch&,            \
                                               const C2<R>*, unsigned long long);                                   \
  template cudaError_t launch_links_from_aos<R, ROWS>(const Geom&, const double*, C2<R>*, cudaStream_t);            \
  template cudaError_t launch_links_to_aos<R, ROWS>(const Geom&, const C2<R>*, double*, cudaStream_t);              \
  template cudaError_t launch_sites_to_aos<R, ROWS>(const Geom&, const C2<R>*, double*, cudaStream_t);              \
  template cudaError_t launch_sites_from_aos<R, ROWS>(const Geom&, const double*, C2<R>*, cudaStream_t);            \
  template cudaError_t launch_set_identity<R, ROWS>(const Geom&, C2<R>*, cudaStream_t);                        \
  template cudaError_t launch_reunitarize_links<R, ROWS>(const Geom&, C2<R>*, DevState*, cudaStream_t);

LGF_INST_R_ROWS(double, 3)
LGF_INST_R_ROWS(double, 2)
LGF_INST_R_ROWS(float, 3)
LGF_INST_R_ROWS(float, 2)

template cudaError_t launch_revert<double, 3, 3>(const Geom&, C2<double>*, const C2<double>*, C2<double>*,
                                                 const DevState*, cudaStream_t, C2<double>*);
template cudaError_t launch_revert<double, 2, 3>(const Geom&, C2<double>*, const C2<double>*, C2<double>*,
                                                 const DevState*, cudaStream_t, C2<double>*);
template cudaError_t launch_revert<float, 2, 2>(const Geom&, C2<float>*, const C2<float>*, C2<float>*,
                                                 const DevState*, cudaStream_t, C2<float>*);
template cudaError_t launch_revert<float, 3, 3>(const Geom&, C2<float>*, const C2<float>*, C2<float>*,
                                                 const DevState*, cudaStream_t, C2<float>*);
template cudaError_t launch_update<double, 3, 3>(const Geom&, C2<double>*, const C2<double>*, const DevState*,
                                                 cudaStream_t, const Batch&);
template cudaError_t launch_update<double, 2, 3>(const Geom&, C2<double>*, const C2<double>*, const DevState*,
                                                 cudaStream_t, const Batch&);
template cudaError_t launch_update<float, 2, 2>(const Geom&, C2<float>*, const C2<float>*, const DevState*,
                                                 cudaStream_t, const Batch&);
template cudaError_t launch_update<float, 3, 3>(const Geom&, C2<float>*, const C2<float>*, const DevState*,
                                                 cudaStream_t, const Batch&);
#define LGF_INST_UM(R, LR, GR)                                                                                     \
  template cudaError_t launch_update_measure<R, LR, GR>(const Geom&, C2<R>*, C2<R>*, const C2<R>*, C2<R>*, double*, \
                                                        DevState*, unsigned long long, int, cudaStream_t,          \
                                                        unsigned long long);
LGF_INST_UM(float, 2, 2)
LGF_INST_UM(float, 3, 3)
template cudaError_t launch_delta_to_aos<double>(const Geom&, const C2<double>*, double*, cudaStream_t);
template cudaError_t launch_delta_to_aos<float>(const Geom&, const C2<float>*, double*, cudaStream_t);
template cudaError_t launch_filter_table<double>(const Geom&, const double*, int, double, double, int, double*,
                                                 cudaStream_t);
template cudaError_t launch_filter_table<float>(const Geom&, const double*, int, double, double, int, float*,
                                                cudaStream_t);

}  // namespace lgf
