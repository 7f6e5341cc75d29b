// The plane passes of FP32 fields on pairs: an element of a tile holds two
// complex values, (re, re) and (im, im), of two fields (x, y) or of two
// neighbouring x columns (z, t), so that one butterfly does both with two-wide
// FP32 instructions and shares its index arithmetic, addresses and twiddles.
//
// The scalar passes of lgf_fft.cu spend about 320 instructions on an element of
// pass B at 48^3x96, a third of them floating point.  Here, besides the pairs,
//   * the first stage of a pass takes its elements from global memory and the
//     last one of pass B stores them there: RAD independent loads per thread and
//     no copy through shared memory of their own;
//   * the last forward stage of pass B, the filter and the first inverse stage
//     act on the same elements and stay in registers.
// 24 x 48 (z, t) planes: 7 trips through shared memory instead of 13, 142
// instructions an element.  A, B, C of 12-real FP32 links, us, scalar -> pairs:
//   16^4       9, 14, 10 -> 8.4, 10.1, 10.1
//   32^4      33, 63, 48 -> 24, 37, 31
//   48^3x96   308, 794, 461 -> 167, 461, 246
// Floors (bytes once at 6.8 TB/s): 10, 10, 12 us at 32^4; 100, 100, 125 us at
// 48^3x96.  What is left is latency: planes of 75 KB leave two CTAs of 384
// threads on an SM, so registers are held to 80 (at 102, one CTA of 512: 277,
// 623, 341 us); pass B of 48^3x96 takes four columns in one CTA of 768 threads
// (runs of 32 bytes; two columns in two CTAs of 384: 507 us).
#include "lgf_fft_tile.cuh"
#include "lgf_gauge.cuh"
#include "lgf_internal.h"

namespace lgf {

// ---------------------------------------------------------------------------
// two-wide arithmetic
// ---------------------------------------------------------------------------

struct CPair {
  float2 re, im;
};
__device__ __forceinline__ float2 two(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return fma2(b, two(-1.f), a); }

__device__ __forceinline__ CPair operator+(CPair a, CPair b) { return CPair{add2(a.re, b.re), add2(a.im, b.im)}; }
__device__ __forceinline__ CPair operator-(CPair a, CPair b) { return CPair{sub2(a.re, b.re), sub2(a.im, b.im)}; }
// a + SIGN i b
template <int SIGN> __device__ __forceinline__ CPair add_i(CPair a, CPair b) {
  return SIGN < 0 ? CPair{add2(a.re, b.im), sub2(a.im, b.re)} : CPair{sub2(a.re, b.im), add2(a.im, b.re)};
}
// a + c b and a + SIGN c i b for real c
__device__ __forceinline__ CPair axpy(float c, CPair b, CPair a) {
  return CPair{fma2(two(c), b.re, a.re), fma2(two(c), b.im, a.im)};
}
template <int SIGN> __device__ __forceinline__ CPair axpy_i(float c, CPair b, CPair a) {
  return CPair{fma2(two(SIGN < 0 ? c : -c), b.im, a.re), fma2(two(SIGN < 0 ? -c : c), b.re, a.im)};
}

// Tile elements and twiddles (w = (cos, cos, -sin, -sin) of the forward root).
__device__ __forceinline__ CPair as_pair(float4 v) { return CPair{make_float2(v.x, v.y), make_float2(v.z, v.w)}; }
__device__ __forceinline__ float4 as_tile(CPair v) { return make_float4(v.re.x, v.re.y, v.im.x, v.im.y); }
template <int SIGN> __device__ __forceinline__ CPair twiddle(CPair v, float4 w) {
  const float2 c = make_float2(w.x, w.y);
  const float2 s = SIGN < 0 ? make_float2(w.z, w.w) : make_float2(-w.z, -w.w);
  const float2 m = SIGN < 0 ? make_float2(-w.z, -w.w) : make_float2(w.z, w.w);
  return CPair{fma2(m, v.im, mul2(c, v.re)), fma2(s, v.re, mul2(c, v.im))};
}

// ---------------------------------------------------------------------------
// DFTs of RAD pairs in registers; SIGN = -1 forward, +1 inverse
// ---------------------------------------------------------------------------

template <int SIGN> __device__ __forceinline__ void dft2(CPair& a, CPair& b) {
  const CPair t = a - b;
  a = a + b;
  b = t;
}
template <int SIGN> __device__ __forceinline__ void dft3(CPair& a, CPair& b, CPair& c) {
  const CPair t = b + c, d = b - c, h = axpy(-0.5f, t, a);
  const float s3 = 0.86602540378443864676372317075294f;  // sin(pi/3)
  a = a + t;
  b = axpy_i<SIGN>(s3, d, h);
  c = axpy_i<-SIGN>(s3, d, h);
}
template <int SIGN> __device__ __forceinline__ void dft4(CPair& a, CPair& b, CPair& c, CPair& d) {
  const CPair p = a + c, m = a - c, q = b + d, n = b - d;
  a = p + q;
  c = p - q;
  b = add_i<SIGN>(m, n);
  d = add_i<-SIGN>(m, n);
}
template <int RAD, int SIGN> __device__ __forceinline__ void dft(CPair* v) {
  if constexpr (RAD == 2) {
    dft2<SIGN>(v[0], v[1]);
  } else if constexpr (RAD == 3) {
    dft3<SIGN>(v[0], v[1], v[2]);
  } else if constexpr (RAD == 4) {
    dft4<SIGN>(v[0], v[1], v[2], v[3]);
  } else if constexpr (RAD == 6) {
    // 2 x 3 without twiddles (Good's mapping): input (3 n1 + 2 n2) mod 6,
    // output (3 k1 + 4 k2) mod 6
    dft2<SIGN>(v[0], v[3]);
    dft2<SIGN>(v[2], v[5]);
    dft2<SIGN>(v[4], v[1]);
    dft3<SIGN>(v[0], v[2], v[4]);
    dft3<SIGN>(v[3], v[5], v[1]);
    const CPair x1 = v[5], x2 = v[4], x4 = v[2], x5 = v[1];
    v[1] = x1;
    v[2] = x2;
    v[4] = x4;
    v[5] = x5;
  } else {
    static_assert(RAD == 8, "radices 2, 3, 4, 6, 8");
    dft4<SIGN>(v[0], v[2], v[4], v[6]);
    dft4<SIGN>(v[1], v[3], v[5], v[7]);
    const CPair e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    const float r = 0.70710678118654752440084436210485f;
    v[0] = e0 + o0;
    v[4] = e0 - o0;
    // e^{SIGN i pi/4} o1 = r (o1 + SIGN i o1), e^{SIGN 3 i pi/4} o3 = r (-o3 + SIGN i o3)
    const CPair p = add_i<SIGN>(o1, o1), m = add_i<-SIGN>(o3, o3);
    v[1] = axpy(r, p, e1);
    v[5] = axpy(-r, p, e1);
    v[2] = add_i<SIGN>(e2, o2);
    v[6] = add_i<-SIGN>(e2, o2);
    v[3] = axpy(-r, m, e3);
    v[7] = axpy(r, m, e3);
  }
}

// ---------------------------------------------------------------------------
// stages over the lines of a tile (the Cooley-Tukey stages of lgf_fft.cu)
// ---------------------------------------------------------------------------

// Butterfly b of a stage: line l, group q = grp Ns + j of the line.
struct Butterfly {
  int l, grp, j;
};
__device__ __forceinline__ Butterfly butterfly(int b, const Lines& ln, const FastDiv& fns) {
  const int q = (int)ln.dn.div((uint32_t)b), grp = (int)fns.div((uint32_t)q);
  return Butterfly{b - q * ln.nlines, grp, q - grp * (int)fns.d};
}
__device__ __forceinline__ int line_base(const Lines& ln, int l) {
  if (ln.inner == ln.nlines) return l * ln.inner_stride;
  const int lo = (int)ln.di.div((uint32_t)l);
  return lo * ln.outer_stride + (l - lo * ln.inner) * ln.inner_stride;
}

template <int RAD, int SIGN> __device__ __forceinline__ void twiddles(CPair* v, int j, int tws, const float4* tw) {
  if (j > 0) {
    const float4* w = tw;
#pragma unroll
    for (int r = 1; r < RAD; ++r) {
      w += j * tws;
      v[r] = twiddle<SIGN>(v[r], *w);
    }
  }
}

template <int RAD, int SIGN, bool DIT>
__device__ __forceinline__ void pair_stage(float4* __restrict__ tile, const Lines& ln, const int N, const FastDiv fns,
                                           const float4* __restrict__ tw) {
  const int Ns = (int)fns.d, nbl = N / RAD, NB = ln.nlines * nbl, tws = nbl / Ns;
  for (int b = threadIdx.x; b < NB; b += blockDim.x) {
    const Butterfly f = butterfly(b, ln, fns);
    float4* p = tile + line_base(ln, f.l) + (f.grp * Ns * RAD + f.j) * ln.es;
    const int step = Ns * ln.es;
    CPair v[RAD];
#pragma unroll
    for (int r = 0; r < RAD; ++r) v[r] = as_pair(p[r * step]);
    if (DIT) twiddles<RAD, SIGN>(v, f.j, tws, tw);
    dft<RAD, SIGN>(v);
    if (!DIT) twiddles<RAD, SIGN>(v, f.j, tws, tw);
#pragma unroll
    for (int r = 0; r < RAD; ++r) p[r * step] = as_tile(v[r]);
  }
  __syncthreads();
}

// Calls f with the radix of a stage as a compile-time number.
template <int N> struct Radix {
  static constexpr int value = N;
};
template <typename F> __device__ __forceinline__ void with_radix(int rad, F&& f) {
  if (rad == 8) f(Radix<8>());
  else if (rad == 4) f(Radix<4>());
  else if (rad == 6) f(Radix<6>());
  else if (rad == 3) f(Radix<3>());
  else f(Radix<2>());
}
template <int SIGN, bool DIT>
__device__ __forceinline__ void pair_stages(float4* tile, const Lines& ln, const FFTDir& d, const float4* tw, int s0,
                                            int s1) {
  for (int k = s0; k < s1; ++k) {
    const int st = DIT ? k : s0 + s1 - 1 - k;
    with_radix(d.radix[st], [&](auto rad) {
      pair_stage<decltype(rad)::value, SIGN, DIT>(tile, ln, d.N, d.ns[st], tw);
    });
  }
}

// Shared memory of a pass: twiddles of two directions, position tables of two
// directions (INV: natural index of a position, otherwise its inverse), tile.
template <bool INV>
__device__ __forceinline__ float4* pair_setup(unsigned char* raw, const float2* __restrict__ twg,
                                              const short* __restrict__ posg, int n0, int n1, float4** tw,
                                              short** pos) {
  *tw = reinterpret_cast<float4*>(raw);
  *pos = reinterpret_cast<short*>(*tw + n0 + n1);
  for (int i = threadIdx.x; i < n0 + n1; i += blockDim.x) {
    const float2 w = __ldg(&twg[i]);
    (*tw)[i] = make_float4(w.x, w.x, w.y, w.y);
    const short p = __ldg(&posg[i]);
    if (INV) (*pos)[(i < n0 ? 0 : n0) + p] = (short)(i < n0 ? i : i - n0);
    else (*pos)[i] = p;
  }
  __syncthreads();
  return reinterpret_cast<float4*>(*pos + ((n0 + n1 + 7) & ~7));
}

static size_t pair_header_bytes(int n0, int n1) {
  return (size_t)(n0 + n1) * sizeof(float4) + (size_t)((n0 + n1 + 7) & ~7) * sizeof(short);
}

// ---------------------------------------------------------------------------
// (x, y) plane pass: one CTA per (z, t) slab and fpb fields, in pairs
// ---------------------------------------------------------------------------

template <int SIGN>
__global__ void __launch_bounds__(PAIR_MAX_THREADS, 2) fft_xy_pair_kernel(Geom g, FFTDir dx, FFTDir dy, float2* __restrict__ data,
                                                          const float2* __restrict__ twg,
                                                          const short* __restrict__ posg, int npp, Lines lx, Lines ly,
                                                          FastDiv dLx, Batch B) {
  if (batch_skip(B)) return;
  data += blockIdx.z * B.s_delta;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int Lx = g.L[0], Ly = g.L[1], RS = Lx | 1, PS = Ly * RS, plane = Lx * Ly;
  float4* tw;
  short* ipos;
  float4* tile = pair_setup<true>(smem_raw, twg, posg, Lx, Ly, &tw, &ipos);
  const int64_t V = g.V;
  float2* fld = data + (int64_t)blockIdx.y * (2 * npp) * V + (int64_t)blockIdx.x * plane;
  // first stage along y from global memory
  with_radix(dy.radix[0], [&](auto rad) {
    constexpr int RAD = decltype(rad)::value;
    const int nbl = Ly / RAD, NB = ly.nlines * nbl;
    for (int b = threadIdx.x; b < NB; b += blockDim.x) {
      const int q = (int)ly.dn.div((uint32_t)b), l = b - q * ly.nlines;
      const int pp = (int)dLx.div((uint32_t)l), px = l - pp * Lx;
      const float2* src = fld + (int64_t)(2 * pp) * V + ipos[Lx + q * RAD] * Lx + ipos[px];
      float2 a[RAD], c[RAD];
#pragma unroll
      for (int r = 0; r < RAD; ++r) {
        a[r] = src[r * nbl * Lx];  // cached: a row's sectors are shared between warps
        c[r] = src[V + r * nbl * Lx];
      }
      CPair v[RAD];
#pragma unroll
      for (int r = 0; r < RAD; ++r) v[r] = CPair{make_float2(a[r].x, c[r].x), make_float2(a[r].y, c[r].y)};
      dft<RAD, SIGN>(v);
      float4* p = tile + pp * PS + q * RAD * RS + px;
#pragma unroll
      for (int r = 0; r < RAD; ++r) p[r * RS] = as_tile(v[r]);
    }
  });
  __syncthreads();
  pair_stages<SIGN, true>(tile, ly, dy, tw + Lx, 1, dy.nst);
  pair_stages<SIGN, true>(tile, lx, dx, tw, 0, dx.nst);
  for (int i = threadIdx.x; i < plane; i += blockDim.x) {
    const int y = (int)dLx.div((uint32_t)i);
    for (int pp = 0; pp < npp; ++pp) {
      const float4 v = tile[pp * PS + i + y * (RS - Lx)];
      fld[(int64_t)(2 * pp) * V + i] = make_float2(v.x, v.z);
      fld[(int64_t)(2 * pp + 1) * V + i] = make_float2(v.y, v.w);
    }
  }
}

// ---------------------------------------------------------------------------
// (z, t) plane pass with the momentum filter: one CTA per (2 xcp x columns, y,
// field).  LRN: the learned handles' variant (multiplier table, divergence
// snapshot).
// ---------------------------------------------------------------------------

// Tile rows (one t): Lz xcp elements, padded so that the eight lanes of a
// 16-byte access that run over neighbouring rows fall on different banks.
static int zt_row(int Lz, int xcp) { return xcp == 1 ? Lz | 1 : Lz * xcp + (((xcp - Lz * xcp) % 8) + 8) % 8; }

template <bool LRN>
__global__ void __launch_bounds__(PAIR_ZT_THREADS) fft_zt_pair_kernel(Geom g, FFTDir dz, FFTDir dt, float2* __restrict__ data,
                                                          const float2* __restrict__ twg,
                                                          const short* __restrict__ posg,
                                                          const float* __restrict__ K, int xcp, int TS, LearnedIO lio,
                                                          int4 H, Lines lz, Lines lt, FastDiv dxcp, FastDiv dxb,
                                                          Batch B) {
  if (batch_skip(B)) return;
  data += blockIdx.z * B.s_delta;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int Lx = g.L[0], Ly = g.L[1], Lz = g.L[2], Lt = g.L[3];
  float4* tw;
  short* ipos;
  float4* tile = pair_setup<true>(smem_raw, twg + Lx + Ly, posg + Lx + Ly, Lz, Lt, &tw, &ipos);
  const int y = (int)dxb.div(blockIdx.x), x0 = ((int)blockIdx.x - y * (int)dxb.d) * 2 * xcp;
  const int64_t plane = (int64_t)Lx * Ly, sxy = (int64_t)y * Lx + x0;
  float2* fld = data + (int64_t)blockIdx.y * g.V + sxy;
  // first forward stage along z from global memory: position grp RAD + r of a
  // z line holds z = ipos[grp RAD] + r Lz / RAD
  with_radix(dz.radix[0], [&](auto rad) {
    constexpr int RAD = decltype(rad)::value;
    const int nbl = Lz / RAD, NB = lz.nlines * nbl;
    for (int b = threadIdx.x; b < NB; b += blockDim.x) {
      const int q = (int)lz.dn.div((uint32_t)b), l = b - q * lz.nlines;
      const int pt = (int)dxcp.div((uint32_t)l), xi = l - pt * xcp;
      const float2* src = fld + (int64_t)(ipos[Lz + pt] * Lz + ipos[q * RAD]) * plane + 2 * xi;
      CPair v[RAD];
#pragma unroll
      for (int r = 0; r < RAD; ++r) {
        const float4 a = __ldcg(reinterpret_cast<const float4*>(src + r * nbl * plane));
        v[r] = CPair{make_float2(a.x, a.z), make_float2(a.y, a.w)};
      }
      dft<RAD, -1>(v);
      float4* p = tile + pt * TS + q * RAD * xcp + xi;
#pragma unroll
      for (int r = 0; r < RAD; ++r) p[r * xcp] = as_tile(v[r]);
    }
  });
  __syncthreads();
  pair_stages<-1, true>(tile, lz, dz, tw, 1, dz.nst);
  pair_stages<-1, true>(tile, lt, dt, tw + Lz, 0, dt.nst - 1);
  // last forward stage along t, the filter and the first inverse stage.
  // learned multiplier of the momentum class (f_mu = min(k_mu, L_mu - k_mu))
  // and the snapshot of the transformed divergence, both of step k
  const int kit = LRN ? lio.st->iter : 0;
  const bool learned = LRN && lio.mtab != nullptr && lio.st->use_m != 0;
  const float* mtab = lio.mtab + (int64_t)(kit & 1) * lio.nclass;
  uint32_t* snap = (LRN && lio.snap != nullptr) ? lio.snap + ((int64_t)(kit & 1) * 4 + blockIdx.y) * g.V : nullptr;
  with_radix(dt.radix[dt.nst - 1], [&](auto rad) {
    constexpr int RAD = decltype(rad)::value;
    const int Ns = Lt / RAD, NB = lt.nlines * Ns;
    for (int b = threadIdx.x; b < NB; b += blockDim.x) {
      const int j = (int)lt.dn.div((uint32_t)b), l = b - j * lt.nlines;
      const int z = (int)dxcp.div((uint32_t)l), xi = l - z * xcp;
      const int64_t k0 = (int64_t)(j * Lz + z) * plane + sxy + 2 * xi, ks = (int64_t)Ns * Lz * plane;
      float2 k[RAD];
#pragma unroll
      for (int r = 0; r < RAD; ++r) k[r] = __ldg(reinterpret_cast<const float2*>(K + k0 + r * ks));
      float4* p = tile + l + j * TS;
      CPair v[RAD];
#pragma unroll
      for (int r = 0; r < RAD; ++r) v[r] = as_pair(p[r * Ns * TS]);
      twiddles<RAD, -1>(v, j, 1, tw + Lz);
      dft<RAD, -1>(v);
#pragma unroll
      for (int r = 0; r < RAD; ++r) {
        if (learned) {
          const int kx = x0 + 2 * xi, t = j + r * Ns;
          const float* m = mtab + ((int64_t)(min(t, Lt - t) * H.z + min(z, Lz - z)) * H.y + min(y, Ly - y)) * H.x;
          k[r].x *= __ldg(m + min(kx, Lx - kx));
          k[r].y *= __ldg(m + min(kx + 1, Lx - kx - 1));
        }
        if (LRN && snap != nullptr) {
          snap[k0 + r * ks] = bf16x2_of<float>(make_float2(v[r].re.x, v[r].im.x));
          snap[k0 + r * ks + 1] = bf16x2_of<float>(make_float2(v[r].re.y, v[r].im.y));
        }
        v[r] = CPair{mul2(v[r].re, k[r]), mul2(v[r].im, k[r])};
      }
      dft<RAD, +1>(v);
      twiddles<RAD, +1>(v, j, 1, tw + Lz);
#pragma unroll
      for (int r = 0; r < RAD; ++r) p[r * Ns * TS] = as_tile(v[r]);
    }
  });
  __syncthreads();
  pair_stages<+1, false>(tile, lt, dt, tw + Lz, 0, dt.nst - 1);
  pair_stages<+1, false>(tile, lz, dz, tw, 1, dz.nst);
  with_radix(dz.radix[0], [&](auto rad) {
    constexpr int RAD = decltype(rad)::value;
    const int nbl = Lz / RAD, NB = lz.nlines * nbl;
    for (int b = threadIdx.x; b < NB; b += blockDim.x) {
      const int q = (int)lz.dn.div((uint32_t)b), l = b - q * lz.nlines;
      const int pt = (int)dxcp.div((uint32_t)l), xi = l - pt * xcp;
      const float4* p = tile + pt * TS + q * RAD * xcp + xi;
      CPair v[RAD];
#pragma unroll
      for (int r = 0; r < RAD; ++r) v[r] = as_pair(p[r * xcp]);
      dft<RAD, +1>(v);
      float2* dst = fld + (int64_t)(ipos[Lz + pt] * Lz + ipos[q * RAD]) * plane + 2 * xi;
#pragma unroll
      for (int r = 0; r < RAD; ++r)
        *reinterpret_cast<float4*>(dst + r * nbl * plane) =
            make_float4(v[r].re.x, v[r].im.x, v[r].re.y, v[r].im.y);
    }
  });
}

// ---------------------------------------------------------------------------
// inverse (x, y) plane pass with g(x)
// ---------------------------------------------------------------------------

template <int GROWS, bool EXPG>
__global__ void __launch_bounds__(PAIR_MAX_THREADS, 2) fft_xy_inv_gauge_pair_kernel(Geom g, FFTDir dx, FFTDir dy,
                                                                    const float2* __restrict__ data,
                                                                    const float2* __restrict__ twg,
                                                                    const short* __restrict__ posg,
                                                                    float2* __restrict__ gf, float2* __restrict__ Gf,
                                                                    Lines lx, Lines ly, FastDiv dLx, Batch B) {
  if (batch_skip(B)) return;
  data += blockIdx.z * B.s_delta;
  gf += blockIdx.z * B.s_g;
  if (Gf != nullptr) Gf += blockIdx.z * B.s_G;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int Lx = g.L[0], Ly = g.L[1], RS = Lx | 1, PS = Ly * RS, plane = Lx * Ly;
  float4* tw;
  short* pos;
  float4* tile = pair_setup<false>(smem_raw, twg, posg, Lx, Ly, &tw, &pos);
  const int64_t V = g.V, s0 = (int64_t)blockIdx.x * plane;
  const float2* fld = data + s0;
  // first inverse stage along y from global memory
  with_radix(dy.radix[dy.nst - 1], [&](auto rad) {
    constexpr int RAD = decltype(rad)::value;
    const int Ns = Ly / RAD, NB = ly.nlines * Ns;
    for (int b = threadIdx.x; b < NB; b += blockDim.x) {
      const int j = (int)ly.dn.div((uint32_t)b), l = b - j * ly.nlines;
      const int pp = (int)dLx.div((uint32_t)l), x = l - pp * Lx;
      const float2* src = fld + (int64_t)(2 * pp) * V + j * Lx + x;
      float2 a[RAD], c[RAD];
#pragma unroll
      for (int r = 0; r < RAD; ++r) {
        a[r] = __ldcg(src + r * Ns * Lx);
        c[r] = __ldcg(src + V + r * Ns * Lx);
      }
      CPair v[RAD];
#pragma unroll
      for (int r = 0; r < RAD; ++r) v[r] = CPair{make_float2(a[r].x, c[r].x), make_float2(a[r].y, c[r].y)};
      dft<RAD, +1>(v);
      twiddles<RAD, +1>(v, j, 1, tw + Lx);
      float4* p = tile + pp * PS + j * RS + x;
#pragma unroll
      for (int r = 0; r < RAD; ++r) p[r * Ns * RS] = as_tile(v[r]);
    }
  });
  __syncthreads();
  pair_stages<+1, false>(tile, ly, dy, tw + Lx, 0, dy.nst - 1);
  pair_stages<+1, false>(tile, lx, dx, tw, 0, dx.nst);
  for (int i = threadIdx.x; i < plane; i += blockDim.x) {
    const int y = (int)dLx.div((uint32_t)i), x = i - y * Lx;
    const float4* p = tile + pos[Lx + y] * RS + pos[x];
    const float4 a = p[0], b = p[PS];
    gauge_site<float, float, GROWS, EXPG>(make_float2(a.x, a.z), make_float2(a.y, a.w), make_float2(b.x, b.z),
                                          make_float2(b.y, b.w), V, s0 + i, gf, Gf);
  }
}

// ---------------------------------------------------------------------------
// shared memory and launchers
// ---------------------------------------------------------------------------

size_t pair_smem_xy(const int L[4], int fields) {
  return pair_header_bytes(L[0], L[1]) + (size_t)(fields / 2) * L[1] * (L[0] | 1) * sizeof(float4);
}
size_t pair_smem_zt(const int L[4], int xc) {
  return pair_header_bytes(L[2], L[3]) + (size_t)L[3] * zt_row(L[2], xc / 2) * sizeof(float4);
}

cudaError_t launch_fft_xy_pair(const Geom& g, const FFTPlan& p, float2* data, const float2* tw, const short* pos,
                               int sign, int nfields, int fpb, int threads, cudaStream_t s, const Batch& B) {
  const int Lx = g.L[0], Ly = g.L[1], RS = Lx | 1, npp = fpb / 2;
  const size_t smem = pair_smem_xy(g.L, fpb);
  const dim3 grid((unsigned)(g.L[2] * g.L[3]), (unsigned)(nfields / fpb), (unsigned)B.n);
  const Lines lx = make_lines(npp * Ly, npp * Ly, RS, 0, 1), ly = make_lines(npp * Lx, Lx, 1, Ly * RS, RS);
  const FastDiv dLx = FastDiv::make((uint32_t)Lx);
  cudaError_t e;
  if (sign < 0) {
    if ((e = allow_smem(fft_xy_pair_kernel<-1>, smem)) != cudaSuccess) return e;
    fft_xy_pair_kernel<-1><<<grid, threads, smem, s>>>(g, p.d[0], p.d[1], data, tw, pos, npp, lx, ly, dLx, B);
  } else {
    if ((e = allow_smem(fft_xy_pair_kernel<+1>, smem)) != cudaSuccess) return e;
    fft_xy_pair_kernel<+1><<<grid, threads, smem, s>>>(g, p.d[0], p.d[1], data, tw, pos, npp, lx, ly, dLx, B);
  }
  return cudaGetLastError();
}

cudaError_t launch_fft_zt_pair(const Geom& g, const FFTPlan& p, float2* data, const float2* tw, const short* pos,
                               const float* K, int nfields, cudaStream_t s, const LearnedIO& lio, const Batch& B) {
  const int xcp = p.xc / 2, Lz = g.L[2], Lt = g.L[3], TS = zt_row(Lz, xcp), nxb = g.L[0] / p.xc;
  const size_t smem = p.smem_zt;
  const dim3 grid((unsigned)(nxb * g.L[1]), (unsigned)nfields, (unsigned)B.n);
  const int4 H = make_int4(g.L[0] / 2 + 1, g.L[1] / 2 + 1, g.L[2] / 2 + 1, g.L[3] / 2 + 1);
  const Lines lz = make_lines(Lt * xcp, xcp, 1, TS, xcp), lt = make_lines(Lz * xcp, Lz * xcp, 1, 0, TS);
  const FastDiv dxcp = FastDiv::make((uint32_t)xcp), dxb = FastDiv::make((uint32_t)nxb);
  cudaError_t e;
  if (lio.mtab != nullptr || lio.snap != nullptr) {
    if ((e = allow_smem(fft_zt_pair_kernel<true>, smem)) != cudaSuccess) return e;
    fft_zt_pair_kernel<true><<<grid, p.threads_zt, smem, s>>>(g, p.d[2], p.d[3], data, tw, pos, K, xcp, TS, lio, H, lz,
                                                              lt, dxcp, dxb, B);
  } else {
    if ((e = allow_smem(fft_zt_pair_kernel<false>, smem)) != cudaSuccess) return e;
    fft_zt_pair_kernel<false><<<grid, p.threads_zt, smem, s>>>(g, p.d[2], p.d[3], data, tw, pos, K, xcp, TS, lio, H,
                                                               lz, lt, dxcp, dxb, B);
  }
  return cudaGetLastError();
}

template <int GROWS>
cudaError_t launch_xy_inv_gauge_pair(const Geom& g, const FFTPlan& p, const float2* data, const float2* tw,
                                     const short* pos, float2* gfield, float2* Gfield, cudaStream_t s, const Batch& B,
                                     bool exact_exp) {
  const int Lx = g.L[0], Ly = g.L[1], RS = Lx | 1;
  const size_t smem = p.smem_c;
  const dim3 grid((unsigned)(g.L[2] * g.L[3]), 1, (unsigned)B.n);
  const Lines lx = make_lines(2 * Ly, 2 * Ly, RS, 0, 1), ly = make_lines(2 * Lx, Lx, 1, Ly * RS, RS);
  const FastDiv dLx = FastDiv::make((uint32_t)Lx);
  cudaError_t e;
  if (exact_exp) {
    if ((e = allow_smem(fft_xy_inv_gauge_pair_kernel<GROWS, true>, smem)) != cudaSuccess) return e;
    fft_xy_inv_gauge_pair_kernel<GROWS, true><<<grid, p.threads_c, smem, s>>>(g, p.d[0], p.d[1], data, tw, pos, gfield,
                                                                              Gfield, lx, ly, dLx, B);
  } else {
    if ((e = allow_smem(fft_xy_inv_gauge_pair_kernel<GROWS, false>, smem)) != cudaSuccess) return e;
    fft_xy_inv_gauge_pair_kernel<GROWS, false><<<grid, p.threads_c, smem, s>>>(g, p.d[0], p.d[1], data, tw, pos,
                                                                               gfield, Gfield, lx, ly, dLx, B);
  }
  return cudaGetLastError();
}
template cudaError_t launch_xy_inv_gauge_pair<2>(const Geom&, const FFTPlan&, const float2*, const float2*,
                                                 const short*, float2*, float2*, cudaStream_t, const Batch&, bool);
template cudaError_t launch_xy_inv_gauge_pair<3>(const Geom&, const FFTPlan&, const float2*, const float2*,
                                                 const short*, float2*, float2*, cudaStream_t, const Batch&, bool);

}  // namespace lgf
