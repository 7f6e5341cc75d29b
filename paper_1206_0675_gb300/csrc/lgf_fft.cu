// 4D Fourier transform of the packed divergence as two plane passes
// (the "2D + 2D" decomposition of arXiv:1206.0675 Sec. 3.2), written for
// shared memory instead of cuFFT plus a reorder kernel:
//
//   pass A : forward DFT over each (x, y) plane                     [k3 removed]
//   pass B : forward DFT over (z, t), multiply by the momentum filter,
//            inverse DFT over (z, t)                                [k4 fused]
//   pass C : inverse DFT over (x, y), then g(x) = reunitarize(1 + Delta'(x))
//            (lgf_gauge.cuh), optionally G <- g G                   [k5 fused]
//
// Each 1D transform is an in-place mixed-radix (2, 3, 4, 6, 8) Cooley-Tukey FFT
// in shared memory (see ct_stage).  Consecutive threads work on neighbouring
// lines and every line stride is padded by one element, so the butterflies'
// shared-memory accesses are free of bank conflicts in every direction.
//
// FP64 fields take the integer passes of lgf_fft_fx.cu, FP32 fields the passes
// on pairs of lgf_fft_pair.cu; the scalar passes here remain for the FP32
// planes that leave nothing to pair (an odd x extent, planes of which one fills
// the shared memory, transforms without the filter) and for the other
// decompositions.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <mutex>
#include <vector>

#include "lgf_fft_tile.cuh"
#include "lgf_gauge.cuh"
#include "lgf_internal.h"

namespace lgf {

// ---------------------------------------------------------------------------
// radix-R DFTs in registers; SIGN = -1 forward (e^{-2 pi i nk/R}), +1 inverse
// ---------------------------------------------------------------------------

template <typename R, int SIGN> __device__ __forceinline__ C2<R> mul_i(C2<R> a) {
  // multiply by SIGN * i
  return SIGN < 0 ? mkc<R>(a.y, -a.x) : mkc<R>(-a.y, a.x);
}

template <typename R, int RAD, int SIGN> struct DFT;

template <typename R, int SIGN> struct DFT<R, 2, SIGN> {
  __device__ __forceinline__ static void run(C2<R>* v) {
    const C2<R> a = v[0], b = v[1];
    v[0] = cadd<R>(a, b);
    v[1] = csub<R>(a, b);
  }
};

template <typename R, int SIGN> struct DFT<R, 3, SIGN> {
  __device__ __forceinline__ static void run(C2<R>* v) {
    const R h = (R)0.5, s3 = (R)0.86602540378443864676372317075294;  // cos(pi/3), sin(pi/3)
    const C2<R> t1 = cadd<R>(v[1], v[2]);
    const C2<R> t2 = mkc<R>(fma(-h, t1.x, v[0].x), fma(-h, t1.y, v[0].y));
    const C2<R> d = csub<R>(v[1], v[2]);
    const C2<R> t3 = mul_i<R, SIGN>(mkc<R>(s3 * d.x, s3 * d.y));
    v[0] = cadd<R>(v[0], t1);
    v[1] = cadd<R>(t2, t3);
    v[2] = csub<R>(t2, t3);
  }
};

template <typename R, int SIGN> struct DFT<R, 4, SIGN> {
  __device__ __forceinline__ static void run(C2<R>* v) {
    const C2<R> a = cadd<R>(v[0], v[2]), b = csub<R>(v[0], v[2]);
    const C2<R> c = cadd<R>(v[1], v[3]), d = mul_i<R, SIGN>(csub<R>(v[1], v[3]));
    v[0] = cadd<R>(a, c);
    v[2] = csub<R>(a, c);
    v[1] = cadd<R>(b, d);
    v[3] = csub<R>(b, d);
  }
};

// 2 x 3 without twiddles (Good's mapping): input (3 n1 + 2 n2) mod 6, output
// (3 k1 + 4 k2) mod 6.
template <typename R, int SIGN> struct DFT<R, 6, SIGN> {
  __device__ __forceinline__ static void run(C2<R>* v) {
    C2<R> s[3] = {cadd<R>(v[0], v[3]), cadd<R>(v[2], v[5]), cadd<R>(v[4], v[1])};
    C2<R> d[3] = {csub<R>(v[0], v[3]), csub<R>(v[2], v[5]), csub<R>(v[4], v[1])};
    DFT<R, 3, SIGN>::run(s);
    DFT<R, 3, SIGN>::run(d);
    v[0] = s[0]; v[4] = s[1]; v[2] = s[2];
    v[3] = d[0]; v[1] = d[1]; v[5] = d[2];
  }
};

template <typename R, int SIGN> struct DFT<R, 8, SIGN> {
  __device__ __forceinline__ static void run(C2<R>* v) {
    C2<R> e[4] = {v[0], v[2], v[4], v[6]};
    C2<R> o[4] = {v[1], v[3], v[5], v[7]};
    DFT<R, 4, SIGN>::run(e);
    DFT<R, 4, SIGN>::run(o);
    const R r2 = (R)0.70710678118654752440084436210485;
    // o[k] *= W8^k, W8 = e^{SIGN 2 pi i / 8}
    {
      const C2<R> a = o[1];  // (1 + SIGN i)/sqrt2
      o[1] = SIGN < 0 ? mkc<R>(r2 * (a.x + a.y), r2 * (a.y - a.x)) : mkc<R>(r2 * (a.x - a.y), r2 * (a.y + a.x));
    }
    o[2] = mul_i<R, SIGN>(o[2]);
    {
      const C2<R> a = o[3];  // (-1 + SIGN i)/sqrt2
      o[3] = SIGN < 0 ? mkc<R>(r2 * (a.y - a.x), -r2 * (a.x + a.y)) : mkc<R>(-r2 * (a.x + a.y), r2 * (a.x - a.y));
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[k] = cadd<R>(e[k], o[k]);
      v[k + 4] = csub<R>(e[k], o[k]);
    }
  }
};

// ---------------------------------------------------------------------------
// in-place mixed-radix Cooley-Tukey stages over a set of lines of a tile
// ---------------------------------------------------------------------------
//
// With radices R_0..R_{m-1} (stage s spans Ns = R_0...R_{s-1}), a butterfly
// of stage s acts on the R_s elements  g*Ns*R_s + j + r*Ns  (r < R_s) of a
// line.  Decimation in time (DIT) multiplies input r by W_{Ns R_s}^{j r}
// before the R_s-point DFT and expects its input in mixed-radix digit-reversed
// order; decimation in frequency (DIF) runs the stages in reverse, applies
// the DFT first and the twiddles to the outputs, and leaves its output in
// digit-reversed order.  The reorder is folded into the global <-> shared
// copies through the position table pos[n] of each direction, so no
// separate reorder kernel (k3 of Sec. 3.2) exists.  A butterfly reads and
// writes only its own elements, so each thread works through its butterflies
// one at a time and stages are separated by a single __syncthreads.

template <typename R, int RAD, int SIGN, bool DIT>
__device__ __forceinline__ void ct_stage(C2<R>* __restrict__ tile, const Lines& ln, const int N, const FastDiv fns,
                                         const C2<R>* __restrict__ tw) {
  const int Ns = (int)fns.d;
  const int nbl = N / RAD;
  const int NB = ln.nlines * nbl;
  const int tws = nbl / Ns;
  for (int b = threadIdx.x; b < NB; b += blockDim.x) {
    const int q = (int)ln.dn.div((uint32_t)b), l = b - q * ln.nlines;
    const int grp = (int)fns.div((uint32_t)q), j = q - grp * Ns;
    const int lo = (int)ln.di.div((uint32_t)l), li = l - lo * ln.inner;
    const int base = lo * ln.outer_stride + li * ln.inner_stride + (grp * Ns * RAD + j) * ln.es;
    const int step = Ns * ln.es;
    C2<R> v[RAD];
#pragma unroll
    for (int r = 0; r < RAD; ++r) v[r] = tile[base + r * step];
    if (DIT && j > 0) {
#pragma unroll
      for (int r = 1; r < RAD; ++r) {
        const C2<R> w = tw[j * r * tws];
        v[r] = SIGN < 0 ? cmul<R>(v[r], w) : cmulc<R>(v[r], w);
      }
    }
    DFT<R, RAD, SIGN>::run(v);
    if (!DIT && j > 0) {
#pragma unroll
      for (int r = 1; r < RAD; ++r) {
        const C2<R> w = tw[j * r * tws];
        v[r] = SIGN < 0 ? cmul<R>(v[r], w) : cmulc<R>(v[r], w);
      }
    }
#pragma unroll
    for (int r = 0; r < RAD; ++r) tile[base + r * step] = v[r];
  }
  __syncthreads();
}

template <typename R, int SIGN, bool DIT>
__device__ __forceinline__ void ct_stage_any(C2<R>* tile, const Lines& ln, int N, const FastDiv& fns, int rad,
                                             const C2<R>* tw) {
  if (rad == 8) ct_stage<R, 8, SIGN, DIT>(tile, ln, N, fns, tw);
  else if (rad == 4) ct_stage<R, 4, SIGN, DIT>(tile, ln, N, fns, tw);
  else if (sizeof(R) == sizeof(float) && rad == 6) ct_stage<R, 6, SIGN, DIT>(tile, ln, N, fns, tw);
  else if (rad == 3) ct_stage<R, 3, SIGN, DIT>(tile, ln, N, fns, tw);
  else ct_stage<R, 2, SIGN, DIT>(tile, ln, N, fns, tw);
}

// DFT of every line: input digit-reversed, output natural.
template <typename R, int SIGN>
__device__ __forceinline__ void fft_lines_dit(C2<R>* tile, const Lines& ln, const FFTDir& d, const C2<R>* tw) {
  for (int st = 0; st < d.nst; ++st) ct_stage_any<R, SIGN, true>(tile, ln, d.N, d.ns[st], d.radix[st], tw);
}

// DFT of every line: input natural, output digit-reversed.
template <typename R, int SIGN>
__device__ __forceinline__ void fft_lines_dif(C2<R>* tile, const Lines& ln, const FFTDir& d, const C2<R>* tw) {
  for (int st = d.nst - 1; st >= 0; --st) ct_stage_any<R, SIGN, false>(tile, ln, d.N, d.ns[st], d.radix[st], tw);
}

// ---------------------------------------------------------------------------
// shared-memory layout helpers
// ---------------------------------------------------------------------------

// Global -> shared copy of one complex element without a register round trip
// (PTX cp.async; 8 bytes for FP32, 16 bytes for FP64, both aligned to their
// size), so that a thread keeps all of its tile's loads in flight at once
// instead of waiting for each before issuing the next.  cp_async_wait() waits
// for this thread's copies; a __syncthreads() after it publishes the tile.
template <typename R> __device__ __forceinline__ void cp_async_elem(C2<R>* dst, const C2<R>* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  if constexpr (sizeof(C2<R>) == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// ---------------------------------------------------------------------------
// (x, y) plane pass: one CTA per (z, t) slab and group of fpb fields;
// digit-reversed load, DIT in x and y, natural store (passes A and, for large
// planes, C).
// ---------------------------------------------------------------------------

template <typename R, int SIGN>
__global__ void __launch_bounds__(512) fft_xy_kernel(Geom g, FFTDir dx, FFTDir dy, C2<R>* __restrict__ data, const C2<R>* __restrict__ twg,
                              const short* __restrict__ posg, int fpb, Lines lx, Lines ly, CopyDiv cd, Batch B) {
  if (batch_skip(B)) return;
  data += blockIdx.z * B.s_delta;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int Lx = g.L[0], Ly = g.L[1];
  C2<R>* tw;
  short* pos;
  C2<R>* tile = setup_smem<R>(smem_raw, twg, posg, Lx, Ly, &tw, &pos);
  const int RS = Lx + 1, PS = Ly * RS;
  const int64_t slab = blockIdx.x;
  const int f0 = blockIdx.y * fpb;
  const int plane = Lx * Ly;
  __syncthreads();
  for (int i = threadIdx.x; i < fpb * plane; i += blockDim.x) {
    const int f = (int)cd.a.div((uint32_t)i), r = i - f * plane, y = (int)cd.b.div((uint32_t)r), x = r - y * Lx;
    cp_async_elem<R>(&tile[f * PS + pos[Lx + y] * RS + pos[x]], &data[(int64_t)(f0 + f) * g.V + slab * plane + r]);
  }
  cp_async_wait();
  __syncthreads();
  fft_lines_dit<R, SIGN>(tile, lx, dx, tw);
  fft_lines_dit<R, SIGN>(tile, ly, dy, tw + Lx);
  for (int i = threadIdx.x; i < fpb * plane; i += blockDim.x) {
    const int f = (int)cd.a.div((uint32_t)i), r = i - f * plane, y = (int)cd.b.div((uint32_t)r), x = r - y * Lx;
    data[(int64_t)(f0 + f) * g.V + slab * plane + r] = tile[f * PS + y * RS + x];
  }
}

// ---------------------------------------------------------------------------
// (z, t) plane pass with the momentum filter: one CTA per (x-block, y, field)
// ---------------------------------------------------------------------------

// LRN: the learned handles' variant (multiplier table, divergence snapshot);
// the plain variant carries none of that code.
template <typename R, bool LRN>
__global__ void __launch_bounds__(512) fft_zt_filter_kernel(Geom g, FFTDir dz, FFTDir dt, C2<R>* __restrict__ data,
                                     const C2<R>* __restrict__ twg, const short* __restrict__ posg,
                                     const R* __restrict__ K, int xc, int mode, LearnedIO lio, int4 H, Lines lz,
                                     Lines lt, CopyDiv cd, Batch B) {
  if (batch_skip(B)) return;
  data += blockIdx.z * B.s_delta;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int Lx = g.L[0], Ly = g.L[1], Lz = g.L[2], Lt = g.L[3];
  C2<R>* tw;
  short* pos;
  C2<R>* tile = setup_smem<R>(smem_raw, twg + Lx + Ly, posg + Lx + Ly, Lz, Lt, &tw, &pos);
  const int TS = Lz * xc + 1;
  const int nxb = Lx / xc;
  const int x0 = (blockIdx.x % nxb) * xc, y = blockIdx.x / nxb;
  C2<R>* fld = data + (int64_t)blockIdx.y * g.V;
  const int n = Lz * Lt * xc;
  const int64_t sxy = (int64_t)y * Lx + x0;
  const int64_t plane = (int64_t)Lx * Ly;
  __syncthreads();
#define LGF_ZT_IDX(i)                                                       \
  const int zt = (int)cd.a.div((uint32_t)(i)), xi = (i) - zt * xc;          \
  const int t = (int)cd.b.div((uint32_t)zt), z = zt - t * Lz;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    LGF_ZT_IDX(i)
    cp_async_elem<R>(&tile[pos[Lz + t] * TS + pos[z] * xc + xi], &fld[(int64_t)zt * plane + sxy + xi]);
  }
  cp_async_wait();
  __syncthreads();
  if (mode == 0) {
    fft_lines_dit<R, -1>(tile, lz, dz, tw);
    fft_lines_dit<R, -1>(tile, lt, dt, tw + Lz);
    // learned multiplier of the momentum class (f_mu = min(k_mu, L_mu - k_mu))
    // and the snapshot of the transformed divergence, both of step k
    const int kit = LRN ? lio.st->iter : 0;
    const bool learned = LRN && lio.mtab != nullptr && lio.st->use_m != 0;
    const float* mtab = lio.mtab + (int64_t)(kit & 1) * lio.nclass;
    uint32_t* snap = (LRN && lio.snap != nullptr) ? lio.snap + ((int64_t)(kit & 1) * 4 + blockIdx.y) * g.V : nullptr;
    const int fy = min(y, Ly - y);
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      LGF_ZT_IDX(i)
      R k = __ldg(&K[(int64_t)zt * plane + sxy + xi]);
      if (learned) {
        const int kx = x0 + xi;
        const int fx = min(kx, Lx - kx), fz = min(z, Lz - z), ft = min(t, Lt - t);
        k *= (R)__ldg(&mtab[((ft * H.z + fz) * H.y + fy) * H.x + fx]);
      }
      C2<R>& e = tile[t * TS + z * xc + xi];
      if (LRN && snap != nullptr) snap[(int64_t)zt * plane + sxy + xi] = bf16x2_of<R>(e);
      e = mkc<R>(e.x * k, e.y * k);
    }
    __syncthreads();
    fft_lines_dif<R, +1>(tile, lt, dt, tw + Lz);
    fft_lines_dif<R, +1>(tile, lz, dz, tw);
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      LGF_ZT_IDX(i)
      fld[(int64_t)zt * plane + sxy + xi] = tile[pos[Lz + t] * TS + pos[z] * xc + xi];
    }
  } else {
    if (mode < 0) {
      fft_lines_dit<R, -1>(tile, lz, dz, tw);
      fft_lines_dit<R, -1>(tile, lt, dt, tw + Lz);
    } else {
      fft_lines_dit<R, +1>(tile, lz, dz, tw);
      fft_lines_dit<R, +1>(tile, lt, dt, tw + Lz);
    }
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      LGF_ZT_IDX(i)
      fld[(int64_t)zt * plane + sxy + xi] = tile[t * TS + z * xc + xi];
    }
  }
#undef LGF_ZT_IDX
}

// ---------------------------------------------------------------------------
// Alternative decompositions of the 4D transform (Sec. 3.2 compares 1D x 4,
// 3D + 1D and 2D + 2D on cuFFT): one pass per direction, or one pass over
// the (x, y, z) slab of each t plus a pass over t.  Both keep every line of a
// pass in shared memory with the same Cooley-Tukey stages as the plane passes.
// ---------------------------------------------------------------------------

// One 1D pass along direction mu.  Contiguous form (mu = x): each CTA takes nl
// consecutive x-lines.  Strided form (mu = y, z, t): each CTA takes xc
// consecutive x columns at fixed other coordinates, so that the global
// accesses are runs of xc elements.  Tile: line l at l * (N + 1).
struct LinePass {
  int N;            // line length L_mu
  int nl;           // lines per CTA
  int contiguous;   // 1 for mu = x
  int64_t S;        // element stride of mu in a field
  int64_t SN;       // S * N
  FastDiv dload;    // by N (contiguous) or by nl (strided)
  FastDiv dlob;     // by S / nl (strided): column blocks per (coordinate above mu)
};

// mode -1: forward DFT; +1: inverse DFT (unnormalised); 0: forward DFT,
// multiplication by K (same layout as the field), inverse DFT.
// mtab (mode 0, may be NULL): learned multiplier per momentum class, applied
// when *use_m != 0; the class of momentum k is (min(k_mu, L_mu - k_mu))_mu in
// a table of H.x * H.y * H.z * H.w classes.
template <typename R, bool LRN>
__global__ void __launch_bounds__(512) fft_line_kernel(LinePass lp, FFTDir d, Geom g, C2<R>* __restrict__ data,
                                                       const C2<R>* __restrict__ twg, const short* __restrict__ posg,
                                                       const R* __restrict__ K, int mode, Lines ln, LearnedIO lio,
                                                       int4 H, Batch B) {
  const int64_t V = g.V;
  if (batch_skip(B)) return;
  data += blockIdx.z * B.s_delta;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2<R>* tw;
  short* pos;
  C2<R>* tile = setup_smem<R>(smem_raw, twg, posg, lp.N, 0, &tw, &pos);
  C2<R>* fld = data + (int64_t)blockIdx.y * V;
  const int N = lp.N, RS = N + 1, n_el = lp.nl * N;
  int64_t s0;
  if (lp.contiguous) {
    s0 = (int64_t)blockIdx.x * n_el;
  } else {
    const uint32_t b = blockIdx.x;
    const uint32_t hi = lp.dlob.div(b), lob = b - hi * lp.dlob.d;
    s0 = (int64_t)lob * lp.nl + (int64_t)hi * lp.SN;
  }
  // element i of the CTA -> (line l, position n) and its site
#define LGF_LINE_IDX(i)                                                          \
  int l, n;                                                                      \
  if (lp.contiguous) { l = (int)lp.dload.div((uint32_t)(i)); n = (i) - l * N; }  \
  else { n = (int)lp.dload.div((uint32_t)(i)); l = (i) - n * lp.nl; }            \
  const int64_t site = lp.contiguous ? s0 + (i) : s0 + l + (int64_t)n * lp.S;
  __syncthreads();
  const bool natural_in = mode > 0;
  for (int i = threadIdx.x; i < n_el; i += blockDim.x) {
    LGF_LINE_IDX(i)
    cp_async_elem<R>(&tile[l * RS + (natural_in ? n : pos[n])], &fld[site]);
  }
  cp_async_wait();
  __syncthreads();
  if (mode < 0) {
    fft_lines_dit<R, -1>(tile, ln, d, tw);
  } else if (mode > 0) {
    fft_lines_dif<R, +1>(tile, ln, d, tw);
  } else {
    fft_lines_dit<R, -1>(tile, ln, d, tw);
    const int kit = LRN ? lio.st->iter : 0;
    const bool learned = LRN && lio.mtab != nullptr && lio.st->use_m != 0;
    const float* mtab = lio.mtab + (int64_t)(kit & 1) * lio.nclass;
    uint32_t* snap = (LRN && lio.snap != nullptr) ? lio.snap + ((int64_t)(kit & 1) * 4 + blockIdx.y) * V : nullptr;
    for (int i = threadIdx.x; i < n_el; i += blockDim.x) {
      LGF_LINE_IDX(i)
      R k = __ldg(&K[site]);
      if (learned) {
        int c[4];
        site_coords(g, site, c);
        const int fx = min(c[0], g.L[0] - c[0]), fy = min(c[1], g.L[1] - c[1]);
        const int fz = min(c[2], g.L[2] - c[2]), ft = min(c[3], g.L[3] - c[3]);
        k *= (R)__ldg(&mtab[((ft * H.z + fz) * H.y + fy) * H.x + fx]);
      }
      C2<R>& e = tile[l * RS + n];
      if (LRN && snap != nullptr) snap[site] = bf16x2_of<R>(e);
      e = mkc<R>(e.x * k, e.y * k);
    }
    __syncthreads();
    fft_lines_dif<R, +1>(tile, ln, d, tw);
  }
  const bool natural_out = mode < 0;
  for (int i = threadIdx.x; i < n_el; i += blockDim.x) {
    LGF_LINE_IDX(i)
    fld[site] = tile[l * RS + (natural_out ? n : pos[n])];
  }
#undef LGF_LINE_IDX
}

// 3D DFT over the (x, y, z) slab of one t and one field (SIGN -1 forward:
// digit-reversed load, DIT, natural store; +1 inverse: natural load, DIF,
// digit-reversed read-out).  The slab must fit in shared memory.
template <typename R, int SIGN>
__global__ void __launch_bounds__(512) fft_xyz_kernel(Geom g, FFTDir dx, FFTDir dy, FFTDir dz, C2<R>* __restrict__ data,
                                                      const C2<R>* __restrict__ twg, const short* __restrict__ posg,
                                                      Lines lx, Lines ly, Lines lz, CopyDiv cd, Batch B) {
  if (batch_skip(B)) return;
  data += blockIdx.z * B.s_delta;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int Lx = g.L[0], Ly = g.L[1], Lz = g.L[2];
  C2<R>* tw;
  short* pos;
  C2<R>* tile = setup_smem<R>(smem_raw, twg, posg, Lx, Ly + Lz, &tw, &pos);
  const int RS = Lx + 1, PS = Ly * RS;
  const int n_el = Lx * Ly * Lz;
  C2<R>* fld = data + (int64_t)blockIdx.y * g.V + (int64_t)blockIdx.x * n_el;
  __syncthreads();
#define LGF_XYZ_IDX(i)                                                     \
  const int z = (int)cd.a.div((uint32_t)(i)), r = (i) - z * Lx * Ly;       \
  const int y = (int)cd.b.div((uint32_t)r), x = r - y * Lx;
  for (int i = threadIdx.x; i < n_el; i += blockDim.x) {
    LGF_XYZ_IDX(i)
    const int o = SIGN < 0 ? pos[Lx + Ly + z] * PS + pos[Lx + y] * RS + pos[x] : z * PS + y * RS + x;
    cp_async_elem<R>(&tile[o], &fld[i]);
  }
  cp_async_wait();
  __syncthreads();
  if (SIGN < 0) {
    fft_lines_dit<R, -1>(tile, lx, dx, tw);
    fft_lines_dit<R, -1>(tile, ly, dy, tw + Lx);
    fft_lines_dit<R, -1>(tile, lz, dz, tw + Lx + Ly);
  } else {
    fft_lines_dif<R, +1>(tile, lz, dz, tw + Lx + Ly);
    fft_lines_dif<R, +1>(tile, ly, dy, tw + Lx);
    fft_lines_dif<R, +1>(tile, lx, dx, tw);
  }
  for (int i = threadIdx.x; i < n_el; i += blockDim.x) {
    LGF_XYZ_IDX(i)
    const int o = SIGN < 0 ? z * PS + y * RS + x : pos[Lx + Ly + z] * PS + pos[Lx + y] * RS + pos[x];
    fld[i] = tile[o];
  }
#undef LGF_XYZ_IDX
}

// ---------------------------------------------------------------------------
// inverse (x, y) plane pass with g(x)
// ---------------------------------------------------------------------------

// Unfused variant for planes whose four fields do not fit in shared memory:
// the inverse (x, y) transform has already been applied to data.
template <typename R, typename RG, int GROWS, bool EXPG>
__global__ void gauge_from_delta_kernel(Geom g, const C2<R>* __restrict__ data, C2<RG>* __restrict__ gf,
                                        C2<RG>* __restrict__ Gf, const DevState* __restrict__ st, Batch B) {
  if (batch_skip(B)) return;
  data += blockIdx.z * B.s_delta;
  gf += blockIdx.z * B.s_g;
  if (Gf != nullptr) Gf += blockIdx.z * B.s_G;
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  gauge_site<R, RG, GROWS, EXPG>(data[s], data[g.V + s], data[2 * g.V + s], data[3 * g.V + s], g.V, s, gf, Gf,
                                 near_identity(st, B));
}

// ---------------------------------------------------------------------------
// plan and launchers
// ---------------------------------------------------------------------------

// Radices of a line of N = 2^a 3^b, as few stages as radices up to 8 allow:
// 16 = 4 x 4 and 128 = 8 x 4 x 4 instead of stages of 2 and, for FP32 fields,
// a left-over 2 or 4 taken into stages of 6 (48 = 8 x 6, 36 = 6 x 6).
static int radix_schedule(int N, int real_bytes, int* radix) {
  int a = 0, b = 0, n = N;
  while (n % 2 == 0) { n /= 2; ++a; }
  while (n % 3 == 0) { n /= 3; ++b; }
  if (n != 1 || N < 2) return -1;
  int k = 0;
  const bool six = real_bytes == 4;
  while (a >= 3 && !(a == 4 && !(six && b > 0))) { radix[k++] = 8; a -= 3; }
  if (a == 4) { radix[k++] = 4; a = 2; }
  while (six && b >= a && a > 0) { radix[k++] = 6; --a; --b; }
  if (a == 2) radix[k++] = 4;
  if (a == 1) radix[k++] = 2;
  while (b-- > 0) radix[k++] = 3;
  return k;
}

// Position of natural index n in the digit-reversed order that the DIT
// stages expect (and the DIF stages produce) for the given radix sequence.
static void digit_positions(int N, const int* radix, int nst, short* pos) {
  if (nst == 0) { pos[0] = 0; return; }
  const int Rl = radix[nst - 1], Ns = N / Rl;
  std::vector<short> sub(Ns);
  digit_positions(Ns, radix, nst - 1, sub.data());
  for (int n = 0; n < N; ++n) pos[n] = (short)((n % Rl) * Ns + sub[n / Rl]);
}

void fft_positions(const FFTPlan& p, short* out) {
  int off = 0;
  for (int mu = 0; mu < 4; ++mu) {
    digit_positions(p.d[mu].N, p.d[mu].radix, p.d[mu].nst, out + off);
    off += p.d[mu].N;
  }
}

static int threads_for(int points) {
  int t = (points + 7) / 8;
  t = ((t + 31) / 32) * 32;
  return std::max(64, std::min(512, t));
}

// Tiles of the 1D x 4 and 3D + 1D decompositions: up to 32 x-lines per CTA
// in the x pass, up to 16 x columns in the y, z, t passes (runs of 16
// elements), and the whole (x, y, z) slab of one field in the 3D pass when
// it fits.
// Tiles of the 1D passes: nl x-lines per CTA in the x pass, xc x columns in
// the y, z, t passes.  False when they do not divide the lattice.
bool set_line_tiles(const int L[4], int real_bytes, int nl, int xc, FFTPlan* p) {
  const size_t cb = 2 * (size_t)real_bytes;
  const int64_t xlines = (int64_t)L[1] * L[2] * L[3];
  if (nl < 1 || xc < 1 || xlines % nl || L[0] % xc) return false;
  p->nl_x = nl;
  p->xc_line = xc;
  for (int mu = 0; mu < 4; ++mu) {
    const int lines = mu == 0 ? nl : xc;
    const size_t hdr = (size_t)((L[mu] + 1) & ~1) * cb + (size_t)((L[mu] + 7) & ~7) * 2;
    p->smem_line[mu] = hdr + (size_t)lines * (L[mu] + 1) * cb;
    p->threads_line[mu] = threads_for(lines * L[mu]);
    if (p->smem_line[mu] > 220 * 1024) return false;
  }
  return true;
}

static void configure_alt_passes(const int L[4], int real_bytes, FFTPlan* p) {
  const size_t cb = 2 * (size_t)real_bytes, maxsm = 220 * 1024;
  const int64_t V = (int64_t)L[0] * L[1] * L[2] * L[3];
  const int64_t xlines = V / L[0];
  int nl = 32;
  while (nl > 1 && (xlines % nl || smem_header_bytes<double>(L[0], 0) + (size_t)nl * (L[0] + 1) * cb > 64 * 1024))
    --nl;
  int xc = 16;
  while (xc > 1 && L[0] % xc) --xc;
  set_line_tiles(L, real_bytes, nl, xc, p);
  const size_t hxyz = (size_t)((L[0] + L[1] + L[2] + 1) & ~1) * cb + (size_t)((L[0] + L[1] + L[2] + 7) & ~7) * 2;
  p->smem_xyz = hxyz + (size_t)L[2] * L[1] * (L[0] + 1) * cb;
  p->fit_xyz = p->smem_xyz <= maxsm ? 1 : 0;
  p->threads_xyz = threads_for(L[0] * L[1] * L[2]);
}

// Shared memory of the plane passes with fpb fields, or xc columns, per CTA.
// FP32 fields go in pairs (lgf_fft_pair.cu) where a CTA has two fields or
// columns to pair.
static bool pairs_xy(int real_bytes, int fields) { return real_bytes == 4 && fields % 2 == 0; }
static bool pairs_zt(int real_bytes, int xc) { return real_bytes == 4 && xc % 2 == 0; }
static size_t xy_smem(const int L[4], int real_bytes, int fields) {
  if (pairs_xy(real_bytes, fields)) return pair_smem_xy(L, fields);
  return plane_header_bytes(L[0], L[1], real_bytes) + (size_t)fields * L[1] * (L[0] + 1) * 2 * real_bytes;
}
static size_t zt_smem(const int L[4], int real_bytes, int xc) {
  if (pairs_zt(real_bytes, xc)) return pair_smem_zt(L, xc);
  return plane_header_bytes(L[2], L[3], real_bytes) + (size_t)L[3] * (L[2] * xc + 1) * 2 * real_bytes;
}

cudaError_t configure_fft_plan(const int L[4], int real_bytes, FFTPlan* p) {
  for (int mu = 0; mu < 4; ++mu) {
    p->d[mu].N = L[mu];
    p->d[mu].nst = radix_schedule(L[mu], real_bytes, p->d[mu].radix);
    if (p->d[mu].nst < 0) return cudaErrorInvalidValue;
    int Ns = 1;
    for (int st = 0; st < p->d[mu].nst; ++st) {
      p->d[mu].ns[st] = FastDiv::make((uint32_t)Ns);
      Ns *= p->d[mu].radix[st];
    }
  }
  const int Lx = L[0], Ly = L[1], Lz = L[2], Lt = L[3];
  const size_t budget = 100 * 1024, maxsm = 220 * 1024;
  // FP64 planes (integer arithmetic, 90 to 130 registers) run best as many
  // small CTAs, one field or one x column each: 412 us for the three passes at
  // 32^4 against 477 us with tiles of 66 KB, and no slower at 16^4 or
  // 24x18x12x27.  FP32 planes take up to four fields and eight columns.
  const bool small = real_bytes == 8;
  p->fpb_xy = small ? 1 : 4;
  while (p->fpb_xy > 1 && xy_smem(L, real_bytes, p->fpb_xy) > (pairs_xy(real_bytes, 2) && p->fpb_xy == 2 ? maxsm : budget))
    p->fpb_xy /= 2;
  p->smem_c = xy_smem(L, real_bytes, 4);
  p->fuse_g = p->smem_c <= (small ? maxsm : PLANE_SMEM_MAX) ? 1 : 0;
  // Planes too large for a fused pass C on few slabs: a field per CTA in the
  // scalar pass, twice as many CTAs.  The three passes, us, pairs -> fields:
  // 96x96x2x4 57 -> 53, 96x96x4x4 64 -> 58, but 96x96x4x8 65 -> 71.
  if (!small && !p->fuse_g && p->fpb_xy == 2 && 4 * Lz * Lt <= 152 / 2 && xy_smem(L, real_bytes, 1) <= budget)
    p->fpb_xy = 1;
  p->smem_xy = xy_smem(L, real_bytes, p->fpb_xy);
  if (p->smem_xy > maxsm) return cudaErrorInvalidValue;
  int xc = 1;
  for (int c = small ? 1 : 8; c >= 1; c /= 2) {
    if (Lx % c) continue;
    if (zt_smem(L, real_bytes, c) <= budget) { xc = c; break; }
  }
  if (!small && xc == 1 && Lx % 2 == 0 && zt_smem(L, real_bytes, 2) <= PLANE_SMEM_MAX) xc = 2;
  // Where only two columns leave room for a second CTA on an SM (runs of 16 bytes,
  // half of each sector), four in one CTA of PAIR_ZT_THREADS.  Pass B, us: 48^3x96
  // 507 -> 461, 64^4 777 -> 651, 16^2x64x96 108 -> 84, 24^2x72x54 127 -> 110.
  const bool alone = !small && xc == 2 && Lx % 4 == 0 && zt_smem(L, real_bytes, 4) <= PLANE_SMEM_MAX;
  if (alone) xc = 4;
  p->xc = xc;
  p->smem_zt = zt_smem(L, real_bytes, xc);
  if (p->smem_zt > (pairs_zt(real_bytes, xc) ? PLANE_SMEM_MAX : maxsm)) return cudaErrorInvalidValue;
  const int most = real_bytes == 8 ? FX_MAX_THREADS : PAIR_MAX_THREADS;
  // Eight elements of a tile per thread (eight pairs where a CTA works on pairs).
  // Lattices of less than two (z, t) slabs per SM take four: an iteration of
  // 16^4 FP32 37.5 -> 34.8 us; the three passes of 32^4 would go 85 -> 93 us.
  const int per = real_bytes == 4 && Lz * Lt < 2 * 152 ? 1 : 2;
  p->threads_xy = std::min(most, threads_for(p->fpb_xy * Lx * Ly / (pairs_xy(real_bytes, p->fpb_xy) ? per : 1)));
  p->threads_zt = std::min(most, threads_for(Lz * Lt * xc / (pairs_zt(real_bytes, xc) ? per : 1)));
  p->threads_c = std::min(most, threads_for(4 * Lx * Ly / (pairs_xy(real_bytes, 4) ? per : 1)));
  if (alone) p->threads_zt = std::min(PAIR_ZT_THREADS, (Lz * Lt * xc / 16 + 31) / 32 * 32);
  if (small && p->fuse_g) {
    // pass C of FP64 planes: as many CTAs as fit an SM's shared memory share its
    // FX_C_THREADS threads (80 registers each).  32^4: three CTAs of 256 110 us,
    // one of 384 threads at 168 registers 150 us, three of 128 126 us;
    // 24x18x12x27 45 -> 31 us.
    const int ctas = std::max(1, (int)(PLANE_SMEM_MAX / (p->smem_c + 1024)));
    p->threads_c = std::min((4 * Lx * Ly / 8 + 31) / 32 * 32, std::max(128, FX_C_THREADS / ctas / 32 * 32));
    p->threads_c = std::max(64, p->threads_c);
  }
  configure_alt_passes(L, real_bytes, p);
  return cudaSuccess;
}

// Candidate plans for the autotuner: the built-in plan, then every
// fields-per-CTA count of the (x,y) passes, every x-column count of the (z,t)
// pass that fits shared memory, and three CTA sizes (8, 16 or 32 elements per
// thread) for each, within the limits of configure_fft_plan.
void fft_plan_candidates(const int L[4], int real_bytes, std::vector<FFTPlan>& out) {
  FFTPlan base;
  out.clear();
  if (configure_fft_plan(L, real_bytes, &base) != cudaSuccess) return;
  out.push_back(base);
  const TuneChoice built_in = tune_choice_of(base, FFT_2D2D);
  const size_t maxsm = 220 * 1024;
  const int Lx = L[0], Ly = L[1], Lz = L[2], Lt = L[3];
  for (int fpb = 1; fpb <= 4; fpb *= 2) {
    if (xy_smem(L, real_bytes, fpb) > maxsm) continue;
    for (int xc = 1; xc <= 8; xc *= 2) {
      const size_t zt = Lx % xc ? 0 : zt_smem(L, real_bytes, xc);
      if (zt == 0 || zt > (pairs_zt(real_bytes, xc) ? PLANE_SMEM_MAX : maxsm)) continue;
      const int most = real_bytes == 8 ? FX_MAX_THREADS : PAIR_MAX_THREADS;
      const int most_zt = pairs_zt(real_bytes, xc) && zt > PLANE_SMEM_MAX / 2 ? PAIR_ZT_THREADS : most;
      for (int tdiv = 8; tdiv <= 32; tdiv *= 2) {
        FFTPlan p = base;
        p.fpb_xy = fpb;
        p.smem_xy = xy_smem(L, real_bytes, fpb);
        p.xc = xc;
        p.smem_zt = zt;
        auto thr = [&](int points, int limit) {
          int t = (points + tdiv - 1) / tdiv;
          t = ((t + 31) / 32) * 32;
          return std::max(64, std::min(limit, t));
        };
        p.threads_xy = thr(fpb * Lx * Ly, most);
        p.threads_zt = thr(Lz * Lt * xc, most_zt);
        p.threads_c = real_bytes == 8 && tdiv == 8 ? base.threads_c : thr(4 * Lx * Ly, most);
        if (!tune_choice_matches(p, built_in)) out.push_back(p);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// autotune cache
// ---------------------------------------------------------------------------

static std::mutex g_tune_mutex;
static std::map<std::string, TuneChoice> g_tune_cache;
static bool g_tune_loaded = false;

TuneChoice tune_choice_of(const FFTPlan& p, int decomp) {
  return TuneChoice{decomp, p.fpb_xy, p.xc, p.threads_xy, p.threads_zt, p.threads_c, p.nl_x, p.xc_line};
}

bool tune_choice_matches(const FFTPlan& p, const TuneChoice& c) {
  return p.fpb_xy == c.fpb_xy && p.xc == c.xc && p.threads_xy == c.threads_xy && p.threads_zt == c.threads_zt &&
         p.threads_c == c.threads_c && p.nl_x == c.nl_x && p.xc_line == c.xc_line;
}

bool tune_cache_get(const std::string& key, TuneChoice* c) {
  std::lock_guard<std::mutex> lock(g_tune_mutex);
  if (!g_tune_loaded) {
    g_tune_loaded = true;
    const char* path = std::getenv("LGF_AUTOTUNE_CACHE");
    FILE* f = path ? std::fopen(path, "r") : nullptr;
    if (f) {
      char k[256];
      TuneChoice t{};
      while (std::fscanf(f, "%255s %d %d %d %d %d %d %d %d", k, &t.decomp, &t.fpb_xy, &t.xc, &t.threads_xy,
                         &t.threads_zt, &t.threads_c, &t.nl_x, &t.xc_line) == 9)
        g_tune_cache[k] = t;
      std::fclose(f);
    }
  }
  auto it = g_tune_cache.find(key);
  if (it == g_tune_cache.end()) return false;
  *c = it->second;
  return true;
}

void tune_cache_put(const std::string& key, const TuneChoice& c) {
  std::lock_guard<std::mutex> lock(g_tune_mutex);
  g_tune_cache[key] = c;
  const char* path = std::getenv("LGF_AUTOTUNE_CACHE");
  FILE* f = path ? std::fopen(path, "a") : nullptr;
  if (!f) return;
  std::fprintf(f, "%s %d %d %d %d %d %d %d %d\n", key.c_str(), c.decomp, c.fpb_xy, c.xc, c.threads_xy, c.threads_zt,
               c.threads_c, c.nl_x, c.xc_line);
  std::fclose(f);
}

template <typename R>
cudaError_t launch_fft_xy(const Geom& g, const FFTPlan& p, C2<R>* data, const C2<R>* tw, const short* pos, int sign,
                          int nfields, cudaStream_t s, const Batch& B) {
  if constexpr (sizeof(R) == sizeof(double)) {
    return launch_fft_xy_fx(g, p, data, tw, pos, sign, nfields, s, B);
  } else {
  int fpb = std::min(p.fpb_xy, nfields);
  while (nfields % fpb) fpb /= 2;
  const int thr = fpb == p.fpb_xy ? p.threads_xy : threads_for(fpb * g.L[0] * g.L[1]);
  if (fpb % 2 == 0)
    return launch_fft_xy_pair(g, p, data, tw, pos, sign, nfields, fpb, std::min(thr, PAIR_MAX_THREADS), s, B);
  const size_t smem = smem_header_bytes<R>(g.L[0], g.L[1]) + (size_t)fpb * g.L[1] * (g.L[0] + 1) * sizeof(C2<R>);
  dim3 grid((unsigned)(g.L[2] * g.L[3]), (unsigned)(nfields / fpb), (unsigned)B.n);
  const int Lx = g.L[0], Ly = g.L[1], RS = Lx + 1, PS = Ly * RS;
  const Lines lx = make_lines(fpb * Ly, fpb * Ly, RS, 0, 1), ly = make_lines(fpb * Lx, Lx, 1, PS, RS);
  const CopyDiv cd{FastDiv::make((uint32_t)(Lx * Ly)), FastDiv::make((uint32_t)Lx)};
  cudaError_t e;
  if (sign < 0) {
    if ((e = allow_smem(fft_xy_kernel<R, -1>, smem)) != cudaSuccess) return e;
    fft_xy_kernel<R, -1><<<grid, thr, smem, s>>>(g, p.d[0], p.d[1], data, tw, pos, fpb, lx, ly, cd, B);
  } else {
    if ((e = allow_smem(fft_xy_kernel<R, +1>, smem)) != cudaSuccess) return e;
    fft_xy_kernel<R, +1><<<grid, thr, smem, s>>>(g, p.d[0], p.d[1], data, tw, pos, fpb, lx, ly, cd, B);
  }
  return cudaGetLastError();
  }
}

template <typename R>
cudaError_t launch_fft_zt(const Geom& g, const FFTPlan& p, C2<R>* data, const C2<R>* tw, const short* pos,
                          const R* K, int mode, int nfields, cudaStream_t s, const LearnedIO& lio, const Batch& B) {
  if constexpr (sizeof(R) == sizeof(double)) {
    return launch_fft_zt_fx(g, p, data, tw, pos, K, mode, nfields, s, lio, B);
  } else {
  if (mode == 0 && p.xc % 2 == 0) return launch_fft_zt_pair(g, p, data, tw, pos, K, nfields, s, lio, B);
  const size_t smem = smem_header_bytes<R>(g.L[2], g.L[3]) + (size_t)g.L[3] * (g.L[2] * p.xc + 1) * sizeof(C2<R>);
  dim3 grid((unsigned)(g.L[0] / p.xc * g.L[1]), (unsigned)nfields, (unsigned)B.n);
  const int threads = std::min(p.threads_zt, 512);  // a plan for pairs can have more
  const bool lrn = mode == 0 && (lio.mtab != nullptr || lio.snap != nullptr);
  cudaError_t e = lrn ? allow_smem(fft_zt_filter_kernel<R, true>, smem) : allow_smem(fft_zt_filter_kernel<R, false>, smem);
  if (e != cudaSuccess) return e;
  const int4 H = make_int4(g.L[0] / 2 + 1, g.L[1] / 2 + 1, g.L[2] / 2 + 1, g.L[3] / 2 + 1);
  const int xc = p.xc, Lz = g.L[2], Lt = g.L[3], TS = Lz * xc + 1;
  const Lines lz = make_lines(Lt * xc, xc, 1, TS, xc), lt = make_lines(Lz * xc, Lz * xc, 1, 0, TS);
  const CopyDiv cd{FastDiv::make((uint32_t)xc), FastDiv::make((uint32_t)Lz)};
  if (lrn)
    fft_zt_filter_kernel<R, true><<<grid, threads, smem, s>>>(g, p.d[2], p.d[3], data, tw, pos, K, p.xc, mode, lio,
                                                                   H, lz, lt, cd, B);
  else
    fft_zt_filter_kernel<R, false><<<grid, threads, smem, s>>>(g, p.d[2], p.d[3], data, tw, pos, K, p.xc, mode,
                                                                    lio, H, lz, lt, cd, B);
  return cudaGetLastError();
  }
}

template <typename R>
cudaError_t launch_fft_line(const Geom& g, const FFTPlan& p, int mu, C2<R>* data, const C2<R>* tw, const short* pos,
                            const R* K, int mode, int nfields, cudaStream_t s, const Batch& B, const LearnedIO& lio) {
  const int N = g.L[mu];
  LinePass lp;
  lp.N = N;
  lp.contiguous = mu == 0;
  lp.nl = mu == 0 ? p.nl_x : p.xc_line;
  lp.S = g.stride[mu];
  lp.SN = lp.S * N;
  lp.dload = FastDiv::make((uint32_t)(lp.contiguous ? N : lp.nl));
  lp.dlob = FastDiv::make((uint32_t)(lp.contiguous ? 1 : lp.S / lp.nl));
  const int64_t blocks = g.V / ((int64_t)N * lp.nl);
  const size_t smem = p.smem_line[mu];
  const bool lrn = mode == 0 && (lio.mtab != nullptr || lio.snap != nullptr);
  cudaError_t e = lrn ? allow_smem(fft_line_kernel<R, true>, smem) : allow_smem(fft_line_kernel<R, false>, smem);
  if (e != cudaSuccess) return e;
  const int off = mu == 0 ? 0 : mu == 1 ? g.L[0] : mu == 2 ? g.L[0] + g.L[1] : g.L[0] + g.L[1] + g.L[2];
  const Lines ln = make_lines(lp.nl, lp.nl, N + 1, 0, 1);
  const int4 H = make_int4(g.L[0] / 2 + 1, g.L[1] / 2 + 1, g.L[2] / 2 + 1, g.L[3] / 2 + 1);
  const dim3 grid((unsigned)blocks, (unsigned)nfields, (unsigned)B.n);
  if (lrn)
    fft_line_kernel<R, true><<<grid, p.threads_line[mu], smem, s>>>(lp, p.d[mu], g, data, tw + off, pos + off, K, mode,
                                                                    ln, lio, H, B);
  else
    fft_line_kernel<R, false><<<grid, p.threads_line[mu], smem, s>>>(lp, p.d[mu], g, data, tw + off, pos + off, K,
                                                                     mode, ln, lio, H, B);
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_fft_xyz(const Geom& g, const FFTPlan& p, C2<R>* data, const C2<R>* tw, const short* pos, int sign,
                           int nfields, cudaStream_t s, const Batch& B) {
  if (!p.fit_xyz) return cudaErrorInvalidConfiguration;
  const int Lx = g.L[0], Ly = g.L[1], Lz = g.L[2], RS = Lx + 1, PS = Ly * RS;
  const Lines lx = make_lines(Ly * Lz, Ly * Lz, RS, 0, 1);
  const Lines ly = make_lines(Lx * Lz, Lx, 1, PS, RS);
  const Lines lz = make_lines(Lx * Ly, Lx, 1, RS, PS);
  const CopyDiv cd{FastDiv::make((uint32_t)(Lx * Ly)), FastDiv::make((uint32_t)Lx)};
  const dim3 grid((unsigned)g.L[3], (unsigned)nfields, (unsigned)B.n);
  cudaError_t e;
  if (sign < 0) {
    if ((e = allow_smem(fft_xyz_kernel<R, -1>, p.smem_xyz)) != cudaSuccess) return e;
    fft_xyz_kernel<R, -1><<<grid, p.threads_xyz, p.smem_xyz, s>>>(g, p.d[0], p.d[1], p.d[2], data, tw, pos, lx, ly, lz,
                                                                  cd, B);
  } else {
    if ((e = allow_smem(fft_xyz_kernel<R, +1>, p.smem_xyz)) != cudaSuccess) return e;
    fft_xyz_kernel<R, +1><<<grid, p.threads_xyz, p.smem_xyz, s>>>(g, p.d[0], p.d[1], p.d[2], data, tw, pos, lx, ly, lz,
                                                                  cd, B);
  }
  return cudaGetLastError();
}

template <typename R, typename RG, int GROWS>
cudaError_t launch_gauge_from_delta(const Geom& g, const C2<R>* data, C2<RG>* gfield, C2<RG>* Gfield,
                                    const DevState* st, cudaStream_t s, const Batch& B, int exact_exp) {
  const dim3 grid((unsigned)((g.V + 127) / 128), 1, (unsigned)B.n);
  if (exact_exp)
    gauge_from_delta_kernel<R, RG, GROWS, true><<<grid, 128, 0, s>>>(g, data, gfield, Gfield, st, B);
  else
    gauge_from_delta_kernel<R, RG, GROWS, false><<<grid, 128, 0, s>>>(g, data, gfield, Gfield, st, B);
  return cudaGetLastError();
}

template <typename R, typename RG, int GROWS, bool EXPG>
static cudaError_t launch_pass_c(const Geom& g, const FFTPlan& p, C2<R>* data, const C2<R>* tw, const short* pos,
                                 C2<RG>* gfield, C2<RG>* Gfield, const DevState* st, cudaStream_t s, const Batch& B) {
  cudaError_t e;
  if (!p.fuse_g) {
    if ((e = launch_fft_xy<R>(g, p, data, tw, pos, +1, 4, s, B)) != cudaSuccess) return e;
    gauge_from_delta_kernel<R, RG, GROWS, EXPG><<<dim3((unsigned)((g.V + 127) / 128), 1, (unsigned)B.n), 128, 0, s>>>(
        g, data, gfield, Gfield, st, B);
    return cudaGetLastError();
  }
  if constexpr (sizeof(R) == sizeof(double)) {
    static_assert(GROWS == 3, "FP64 lanes keep three rows of g");
    return launch_xy_inv_gauge_fx(g, p, data, tw, pos, gfield, Gfield, st, s, B, EXPG);
  } else {
  return launch_xy_inv_gauge_pair<GROWS>(g, p, data, tw, pos, gfield, Gfield, s, B, EXPG);
  }
}

template <typename R, typename RG, int GROWS>
cudaError_t launch_fft_xy_inv_gauge(const Geom& g, const FFTPlan& p, C2<R>* data, const C2<R>* tw, const short* pos,
                                    C2<RG>* gfield, C2<RG>* Gfield, const DevState* st, cudaStream_t s,
                                    const Batch& B, int exact_exp) {
  return exact_exp ? launch_pass_c<R, RG, GROWS, true>(g, p, data, tw, pos, gfield, Gfield, st, s, B)
                   : launch_pass_c<R, RG, GROWS, false>(g, p, data, tw, pos, gfield, Gfield, st, s, B);
}

template cudaError_t launch_fft_xy<double>(const Geom&, const FFTPlan&, C2<double>*, const C2<double>*, const short*,
                                           int, int, cudaStream_t, const Batch&);
template cudaError_t launch_fft_xy<float>(const Geom&, const FFTPlan&, C2<float>*, const C2<float>*, const short*,
                                          int, int, cudaStream_t, const Batch&);
template cudaError_t launch_fft_zt<double>(const Geom&, const FFTPlan&, C2<double>*, const C2<double>*, const short*,
                                           const double*, int, int, cudaStream_t, const LearnedIO&, const Batch&);
template cudaError_t launch_fft_zt<float>(const Geom&, const FFTPlan&, C2<float>*, const C2<float>*, const short*,
                                          const float*, int, int, cudaStream_t, const LearnedIO&, const Batch&);
#define LGF_INST_C(R, RG, GR)                                                                                    \
  template cudaError_t launch_fft_xy_inv_gauge<R, RG, GR>(const Geom&, const FFTPlan&, C2<R>*, const C2<R>*,      \
                                                          const short*, C2<RG>*, C2<RG>*, const DevState*,        \
                                                          cudaStream_t, const Batch&, int);
LGF_INST_C(double, double, 3)
LGF_INST_C(float, float, 2)
LGF_INST_C(float, float, 3)
#define LGF_INST_G(R, RG, GR)                                                                                   \
  template cudaError_t launch_gauge_from_delta<R, RG, GR>(const Geom&, const C2<R>*, C2<RG>*, C2<RG>*,         \
                                                          const DevState*, cudaStream_t, const Batch&, int);
LGF_INST_G(double, double, 3)
LGF_INST_G(double, double, 2)
LGF_INST_G(float, float, 2)
LGF_INST_G(float, float, 3)
#define LGF_INST_ALT(R)                                                                                         \
  template cudaError_t launch_fft_line<R>(const Geom&, const FFTPlan&, int, C2<R>*, const C2<R>*, const short*, \
                                          const R*, int, int, cudaStream_t, const Batch&, const LearnedIO&);   \
  template cudaError_t launch_fft_xyz<R>(const Geom&, const FFTPlan&, C2<R>*, const C2<R>*, const short*, int,  \
                                         int, cudaStream_t, const Batch&);
LGF_INST_ALT(double)
LGF_INST_ALT(float)

}  // namespace lgf
