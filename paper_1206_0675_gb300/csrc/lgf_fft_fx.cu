// The plane passes of the 4D transform for FP64 fields in block floating
// point on the integer pipe.
//
// The FP64 pipe (2 operations per clock and SM) bounds an FP64 Cooley-Tukey
// pass; here a plane is held as 64-bit integers with one exponent, whose
// additions are exact and run on the integer pipe (64 per clock and SM), and
// whose products with twiddles take three 32 x 32 + 64 bit multiply-adds.
//
// Exponents.  A plane of one field gets its own exponent, from the largest
// component of its input, so results do not depend on how planes are grouped
// into CTAs.  A transform of length N is safe from overflow when components
// enter below 2^(61 - h), h = ceil(log2 N) + 1: a sum of N complex terms stays
// below sqrt(2) N 2^(61 - h) <= 2^60.5 in modulus, within the 31-bit upper limb
// of bfp_limbs.  Between the two directions of a plane, and within one of more
// than 64 elements, the largest component is measured again and the plane shifted right by what the next direction
// needs (about half of h for data without structure, so some 55 bits remain
// below the largest component; an FP64 pass keeps 53 bits in each number and
// rounds at every operation, where additions are exact here).  Inputs are
// read and results written in FP64.
//
// Error against extended precision: of the transform (2-norm, forward and
// inverse, random, smooth and constant inputs) 0.7e-16 to 2.8e-16, of the passes
// on the FP64 pipe 1.5e-16 to 4.6e-16; of g(x), where the filter weights the
// lowest modes most (rms): planes of 16 x 16 0.7e-16 (1.1e-16), 32 x 32 1.2e-16
// (1.9e-16), 48 x 48 2.1e-16 (3.0e-16), 64 x 64 5.1e-16 (7.0e-16); longer lines at
// FxCut.  For that every rounding is centred: inputs are rounded, halves go to
// even, and products carry the mean of what they drop.
//
// 32^4, us: pass A 72 (FP64 pipe: 231), pass B 160 (463), pass C with g 110 (397);
// 24x18x12x27: 23, 40, 33 (54, 94, 78).  Bound by latency: about 400 instructions
// per element of pass A, 800 of pass B, at 1.9 to 2.1 a clock and SM of the 4 it
// can issue; the 13 to 20 warps that are active wait on fixed latencies and on
// memory.  80 registers a thread (pass B at 96: 151 us at 32^4, but 53 at 24x18x12x27; at
// 64: 177).
//
// Planes that hold infinities or NaN give NaN; planes whose largest
// component is near the ends of the FP64 range take slower conversions.
#include <algorithm>
#include <cmath>

#include "lgf_fft_tile.cuh"
#include "lgf_fixed.cuh"
#include "lgf_gauge.cuh"
#include "lgf_internal.h"
#include "lgf_roots.h"

namespace lgf {

using I2 = longlong2;

// Per-plane exponents of the (at most 8) planes of a tile, for one transform:
// the largest input component (high word of its magnitude, then the words of
// fx_classify and fx_finish) and, where the plane is measured again (FxCut),
// the bits of its largest component (high word, or-ed).
struct FxTransform {
  uint32_t in[8], mid[3][8];
};
struct FxPlanes {  // a pass holds up to two transforms
  FxTransform t[2];
};
static_assert(sizeof(FxPlanes) == FX_PLANE_BYTES, "header of the FP64 plane passes");

// ceil(log2 N) + 1
static uint32_t fx_headroom(int N) {
  uint32_t h = 1;
  while ((1 << (h - 1)) < N) ++h;
  return h;
}

// The word of a plane after fx_classify: the biased exponent that its input
// is scaled by and, above bit 16, what was done to a plane out of the ordinary:
// scaled up or down by 2^FX_ODD_SCALE so that every exponent that can occur is
// far from the ends of the FP64 range (all-zero planes among them), or set to
// zero because it holds infinities or NaN.
constexpr int FX_ODD_SCALE = 600;
enum { FX_UP = 1, FX_DOWN = 2, FX_NONFINITE = 3 };
__device__ __forceinline__ uint32_t fx_exp_of(uint32_t code) { return code & 0xffffu; }
__device__ __forceinline__ uint32_t fx_classify(uint32_t in) {
  const uint32_t e = max(in >> 20, 1u);
  if (e < 100u) return (e + FX_ODD_SCALE) | (FX_UP << 16);
  if (e == 2047u) return 1023u | (FX_NONFINITE << 16);
  if (e > 1990u) return (e - FX_ODD_SCALE) | (FX_DOWN << 16);
  return e;
}
// Right shift between the directions.
__device__ __forceinline__ uint32_t fx_mid_shift(uint32_t mid, uint32_t h1) {
  const int sh = (64 - __clz((int)mid)) - (int)(61u - h1);
  return (uint32_t)max(sh, 0);
}

// Where the stages of a direction are cut in two, so that the plane is
// measured, and shifted by no more than it needs, between them as well: lines
// of more than 64, whose 8 bits of headroom leave 53 for the largest
// component.  Cut, they enter with 56 or more.  The radices are 8|9, 9|9, 8|12,
// 12|9 and 8|16 for 72 to 128 (decimation in time; in frequency the reverse).
// g(x) of one step, rms in 1e-16, uncut -> cut (passes on the FP64 pipe): planes
// of 72 x 72 10.5 -> 3.1 (8.0), 81 x 81 16.5 -> 5.1 (9.3), 96 x 72 13.7 -> 5.5
// (11.9), 128 x 54 15.2 -> 9.5 (14.7), (z, t) planes of 128 x 81 11.9 -> 5.8 (9.6).
constexpr int FX_CUT_ABOVE = 64;
struct FxCut {
  int first;        // stages before the cut (all of them where there is none)
  uint32_t h0, h1;  // headroom of the two parts
};
static FxCut fx_cut(const FFTDir& d, bool dit) {
  if (d.N <= FX_CUT_ABOVE) return FxCut{d.nst, fx_headroom(d.N), 0u};
  const int q = (int)d.ns[d.nst - 2].d;  // the product of all radices but the last two
  const uint32_t ha = fx_headroom(q), hb = fx_headroom(d.N / q);
  return dit ? FxCut{d.nst - 2, ha, hb} : FxCut{2, hb, ha};
}

// The stages of a plane transform in order, made on the host, so that a kernel
// reads from constant memory what each stage does and keeps no state of its own
// (registers bound these kernels).  A step: axis, stage of the axis from bit 4,
// headroom of its part of the direction from bit 8; bit 16: raw FP64 input,
// scaled by FxTransform::in; from bit 20, m > 0: integers to be shifted by what
// mid[m - 1] measured; from bit 24, m > 0: record the bits of the outputs in
// mid[m - 1]; bit 28: the last stage.
struct FxProgram {
  int n;
  uint32_t step[16];
  uint32_t h[3], h0;  // headroom behind each measurement (0: none), and of the first stages
};
static FxProgram fx_program(const FFTDir d[2], int first, bool dit) {
  FxProgram P{};
  for (int k = 0; k < 2; ++k) {
    const int ax = first ^ k;
    const FxCut c = fx_cut(d[ax], dit);
    for (int i = 0; i < d[ax].nst; ++i) {
      const bool start = i == 0, cut = i == c.first, end = i == d[ax].nst - 1;
      const uint32_t h = i < c.first ? c.h0 : c.h1;
      const uint32_t shift = cut ? 2 * k + 1 : start && k == 1 ? 2 : 0;
      const uint32_t mid = end ? (k == 0 ? 2 : 0) : i == c.first - 1 ? 2 * k + 1 : 0;
      const uint32_t st = (uint32_t)(dit ? i : d[ax].nst - 1 - i);
      P.step[P.n++] = (uint32_t)ax | st << 4 | h << 8 | (uint32_t)(start && k == 0) << 16 | shift << 20 | mid << 24 |
                      (uint32_t)(end && k == 1) << 28;
      if (shift) P.h[shift - 1] = h;
    }
    if (k == 0) P.h0 = c.h0;
  }
  return P;
}

__device__ __forceinline__ I2 fx_in(double2 v, uint32_t base) {
  return make_longlong2(bfp_from(v.x, base), bfp_from(v.y, base));
}

// The word of a plane after its transform: the exponent of its integers (of the
// scaled plane) and the class of fx_classify.
__device__ __forceinline__ uint32_t fx_finish(const FxTransform* t, int pl, const FxProgram& P) {
  const uint32_t code = t->in[pl];
  uint32_t sh = fx_mid_shift(t->mid[1][pl], P.h[1]);
  if (P.h[0] != 0u) sh += fx_mid_shift(t->mid[0][pl], P.h[0]);
  if (P.h[2] != 0u) sh += fx_mid_shift(t->mid[2][pl], P.h[2]);
  return (code & 0xffff0000u) | (sh + P.h0 + fx_exp_of(code) - 1083u + 4096u);
}
__device__ __forceinline__ int fx_out_exp(uint32_t word) { return (int)(word & 0xffffu) - 4096; }
// The exponent of the plane as it was, large where it holds infinities or NaN.
__device__ __forceinline__ int fx_true_exp(uint32_t word) {
  const int ex = fx_out_exp(word);
  const uint32_t k = word >> 16;
  return k == 0u ? ex : k == FX_UP ? ex - FX_ODD_SCALE : k == FX_DOWN ? ex + FX_ODD_SCALE : 4096;
}
// Output of a plane after both directions.
__device__ __forceinline__ double2 fx_out(I2 v, uint32_t word) {
  const int ex = fx_out_exp(word);
  return make_double2(bfp_to_double(v.x, ex), bfp_to_double(v.y, ex));
}
// The same for any plane.
static __device__ __noinline__ double2 fx_out_any(I2 v, uint32_t word) {
  if (word >> 16 == FX_NONFINITE) return make_double2(NAN, NAN);
  const double2 r = fx_out(v, word);
  const int k = word >> 16 == FX_UP ? -FX_ODD_SCALE : word >> 16 == FX_DOWN ? FX_ODD_SCALE : 0;
  return make_double2(scalbn(r.x, k), scalbn(r.y, k));
}

// v 2^ex in units of 2^-58, rounded; ok = false unless it is below 1 in magnitude.
__device__ __forceinline__ int64_t fx_unit58(int64_t v, int ex, bool& ok) {
  if (ex > -62) {  // |v| 2^ex can reach 1
    const uint64_t u = (uint64_t)(v ^ (v >> 63));
    ok = ok && ex < 0 && shr64_clamp(u, (uint32_t)-ex) == 0;
  }
  const int sh = -58 - ex;
  if (sh <= 0) return (int64_t)((uint64_t)v << (-sh & 63));
  const int c = min(sh, 63);
  return (v + ((int64_t)1 << (c - 1))) >> c;
}

struct FxOut {
  __device__ __forceinline__ double2 operator()(I2 v, uint32_t word) const { return fx_out(v, word); }
};
struct FxOutAny {
  __device__ __forceinline__ double2 operator()(I2 v, uint32_t word) const { return fx_out_any(v, word); }
};

__device__ __forceinline__ I2 iadd(I2 a, I2 b) { return make_longlong2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ I2 isub(I2 a, I2 b) { return make_longlong2(a.x - b.x, a.y - b.y); }
// v >> s (s >= 1), ties to even: a bias would add up in the zero mode.
__device__ __forceinline__ int64_t ishift(int64_t v, uint32_t s) {
  return (v + ((int64_t)1 << (s - 1)) - 1 + ((v >> s) & 1)) >> s;
}
template <int SIGN> __device__ __forceinline__ I2 imul_i(I2 a) {  // times SIGN i
  return SIGN < 0 ? make_longlong2(a.y, -a.x) : make_longlong2(-a.y, a.x);
}

// v w (SIGN < 0) or v conj(w) for a table entry w = (cos h, l, sin h, l).
template <int SIGN> __device__ __forceinline__ I2 itwiddle(I2 v, int4 w) {
  const Bfp2 x = bfp_limbs(v.x), y = bfp_limbs(v.y);
  const int sh = fx_opaque(SIGN < 0 ? w.z : -w.z), sl = fx_opaque(SIGN < 0 ? w.w : -w.w);
  const int nh = fx_opaque(SIGN < 0 ? -w.z : w.z), nl = fx_opaque(SIGN < 0 ? -w.w : w.w);
  const int64_t half = (int64_t)1 << 29;  // and the mean of the products of low limbs (bfp_mul)
  int64_t rm = mad_wide(x.l, w.x, mad_wide(x.h, w.y, half + ((w.y + nl) >> 1)));
  int64_t im = mad_wide(x.l, sh, mad_wide(x.h, sl, half + ((sl + w.y) >> 1)));
  rm = mad_wide(y.l, nh, mad_wide(y.h, nl, rm));
  im = mad_wide(y.l, w.x, mad_wide(y.h, w.y, im));
  return make_longlong2(mad_wide(y.h, nh, mad_wide(x.h, w.x, rm >> 30)),
                        mad_wide(y.h, w.x, mad_wide(x.h, sh, im >> 30)));
}

// 1/sqrt 2 and sqrt(3)/2 as h 2^-30 + l 2^-60
constexpr int IR2_H = 759250125, IR2_L = -6429112;
constexpr int IS3_H = 929887697, IS3_L = -333032134;

template <int RAD, int SIGN> struct IDFT;
template <int SIGN> struct IDFT<2, SIGN> {
  __device__ __forceinline__ static void run(I2* v) {
    const I2 a = v[0], b = v[1];
    v[0] = iadd(a, b);
    v[1] = isub(a, b);
  }
};
template <int SIGN> struct IDFT<3, SIGN> {
  __device__ __forceinline__ static void run(I2* v) {
    const I2 t1 = iadd(v[1], v[2]);
    const I2 t2 = make_longlong2(v[0].x - ishift(t1.x, 1), v[0].y - ishift(t1.y, 1));
    const I2 d = isub(v[1], v[2]);
    const I2 t3 = imul_i<SIGN>(make_longlong2(bfp_mul(d.x, IS3_H, IS3_L), bfp_mul(d.y, IS3_H, IS3_L)));
    v[0] = iadd(v[0], t1);
    v[1] = iadd(t2, t3);
    v[2] = isub(t2, t3);
  }
};
template <int SIGN> struct IDFT<4, SIGN> {
  __device__ __forceinline__ static void run(I2* v) {
    const I2 a = iadd(v[0], v[2]), b = isub(v[0], v[2]);
    const I2 c = iadd(v[1], v[3]), d = imul_i<SIGN>(isub(v[1], v[3]));
    v[0] = iadd(a, c);
    v[2] = isub(a, c);
    v[1] = iadd(b, d);
    v[3] = isub(b, d);
  }
};
template <int SIGN> struct IDFT<8, SIGN> {
  __device__ __forceinline__ static void run(I2* v) {
    I2 e[4] = {v[0], v[2], v[4], v[6]};
    I2 o[4] = {v[1], v[3], v[5], v[7]};
    IDFT<4, SIGN>::run(e);
    IDFT<4, SIGN>::run(o);
    {  // times (1 + SIGN i)/sqrt 2
      const I2 a = o[1];
      const int64_t p = bfp_mul(a.x + a.y, IR2_H, IR2_L), q = bfp_mul(a.y - a.x, IR2_H, IR2_L);
      o[1] = SIGN < 0 ? make_longlong2(p, q) : make_longlong2(-q, p);
    }
    o[2] = imul_i<SIGN>(o[2]);
    {  // times (-1 + SIGN i)/sqrt 2
      const I2 a = o[3];
      const int64_t p = bfp_mul(a.x + a.y, IR2_H, IR2_L), q = bfp_mul(a.y - a.x, IR2_H, IR2_L);
      o[3] = SIGN < 0 ? make_longlong2(q, -p) : make_longlong2(-p, -q);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[k] = iadd(e[k], o[k]);
      v[k + 4] = isub(e[k], o[k]);
    }
  }
};

// One stage, as ct_stage of lgf_fft.cu; io: the step of FxProgram.  The plane of line l is l / inner
// (PLO) or l % inner.
template <int RAD, int SIGN, bool DIT, bool PLO>
__device__ __forceinline__ void fx_stage(I2* __restrict__ tile, const Lines& ln, const int N, const FastDiv fns,
                                         const int4* __restrict__ tw, const uint32_t io, FxTransform* t) {
  const int Ns = (int)fns.d;
  const int nbl = N / RAD;
  const int NB = ln.nlines * nbl;
  const int tws = nbl / Ns;
  for (int b = threadIdx.x; b < NB; b += blockDim.x) {
    const int q = (int)ln.dn.div((uint32_t)b), l = b - q * ln.nlines;
    const int grp = (int)fns.div((uint32_t)q), j = q - grp * Ns;
    const int lo = (int)ln.di.div((uint32_t)l), li = l - lo * ln.inner;
    const int pl = PLO ? lo : li;
    const int base = lo * ln.outer_stride + li * ln.inner_stride + (grp * Ns * RAD + j) * ln.es;
    const int step = Ns * ln.es;
    I2 v[RAD];
    if (io & (1u << 16)) {
      const double2* raw = reinterpret_cast<const double2*>(tile);
      const uint32_t sc = 3u + ((io >> 8) & 15u) + fx_exp_of(t->in[pl]);
#pragma unroll
      for (int r = 0; r < RAD; ++r) v[r] = fx_in(raw[base + r * step], sc);
    } else {
#pragma unroll
      for (int r = 0; r < RAD; ++r) v[r] = tile[base + r * step];
      if (io & (3u << 20)) {
        const uint32_t sh = fx_mid_shift(t->mid[((io >> 20) & 3u) - 1u][pl], (io >> 8) & 15u);
        if (sh != 0u) {
#pragma unroll
          for (int r = 0; r < RAD; ++r) v[r] = make_longlong2(ishift(v[r].x, sh), ishift(v[r].y, sh));
        }
      }
    }
    if (DIT && j > 0) {
#pragma unroll
      for (int r = 1; r < RAD; ++r) v[r] = itwiddle<SIGN>(v[r], tw[j * r * tws]);
    }
    IDFT<RAD, SIGN>::run(v);
    if (!DIT && j > 0) {
#pragma unroll
      for (int r = 1; r < RAD; ++r) v[r] = itwiddle<SIGN>(v[r], tw[j * r * tws]);
    }
#pragma unroll
    for (int r = 0; r < RAD; ++r) tile[base + r * step] = v[r];
    if (io & (3u << 24)) {
      uint32_t* mid = t->mid[((io >> 24) & 3u) - 1u];
      uint32_t m = 0;
#pragma unroll
      for (int r = 0; r < RAD; ++r) {
        m |= (uint32_t)(v[r].x >> 32) ^ (uint32_t)(v[r].x >> 63);
        m |= (uint32_t)(v[r].y >> 32) ^ (uint32_t)(v[r].y >> 63);
      }
      if (PLO) {
        // the lanes of a warp mostly share a plane: one atomic for all of them
        const unsigned act = __activemask();
        const int lead = __ffs((int)act) - 1;
        if (__all_sync(act, pl == __shfl_sync(act, pl, lead))) {
          m = __reduce_or_sync(act, m);
          if ((int)(threadIdx.x & 31) == lead) atomicOr(&mid[pl], m);
        } else {
          atomicOr(&mid[pl], m);
        }
      } else {
        atomicOr(&mid[pl], m);
      }
    }
  }
  __syncthreads();
}

// The two directions of a plane pass: d[0] and l[0] the first axis of the
// plane (x or z), d[1] and l[1] the second.
struct FxPass {
  FFTDir d[2];
  Lines l[2];
  FxProgram p[2];  // its transforms, in order
};

// Both directions of a plane transform from raw FP64 input; DIT takes
// digit-reversed input and gives natural order, DIF the reverse.  One loop over
// the stages of both: those of a radix are the same code (the instruction cache
// held neither copy otherwise).  Leaves the word of each plane (fx_finish) in
// t->in; ends with a __syncthreads.
template <int SIGN, bool DIT, bool PLO>
__device__ __forceinline__ void fx_plane(I2* tile, const FxPass& P, const FxProgram& prog, const int4* tw, int nplanes,
                                         FxTransform* t) {
#pragma unroll 1
  for (int i = 0; i < prog.n; ++i) {
    const uint32_t io = prog.step[i];
    const int ax = (int)(io & 1u), st = (int)(io >> 4) & 15;
    const FFTDir& d = P.d[ax];
    const Lines& ln = P.l[ax];
    const int4* w = ax == 0 ? tw : tw + P.d[0].N;
    // every measurement is complete before the last stage
    if (io >> 28 && (int)threadIdx.x < nplanes) t->in[threadIdx.x] = fx_finish(t, threadIdx.x, prog);
    if (d.radix[st] == 8) fx_stage<8, SIGN, DIT, PLO>(tile, ln, d.N, d.ns[st], w, io, t);
    else if (d.radix[st] == 4) fx_stage<4, SIGN, DIT, PLO>(tile, ln, d.N, d.ns[st], w, io, t);
    else if (d.radix[st] == 3) fx_stage<3, SIGN, DIT, PLO>(tile, ln, d.N, d.ns[st], w, io, t);
    else fx_stage<2, SIGN, DIT, PLO>(tile, ln, d.N, d.ns[st], w, io, t);
  }
}

// Tile of a plane pass: header as setup_smem, then the plane exponents.
__device__ __forceinline__ I2* fx_setup(unsigned char* raw, const int4* __restrict__ twg, const short* __restrict__ posg,
                                        int n0, int n1, int4** tw, short** pos, FxPlanes** ps) {
  double2* t2;
  double2* after = setup_smem<double>(raw, reinterpret_cast<const double2*>(twg), posg, n0, n1, &t2, pos);
  *tw = reinterpret_cast<int4*>(t2);
  *ps = reinterpret_cast<FxPlanes*>(after);
  if (threadIdx.x < FX_PLANE_BYTES / 4) reinterpret_cast<uint32_t*>(*ps)[threadIdx.x] = 0u;
  return reinterpret_cast<I2*>(*ps + 1);
}

// Copies n elements global -> tile (src(i), dst(i), plane(i)), recording the
// largest component of every plane; four loads in flight per thread.
template <typename SRC, typename DST>
__device__ __forceinline__ void fx_load(I2* tile, int n, uint32_t* in, SRC src, DST dst) {
  double2* raw = reinterpret_cast<double2*>(tile);
  int cur = -1;
  uint32_t m = 0;
  for (int i0 = threadIdx.x; i0 < n; i0 += 4 * blockDim.x) {
    double2 v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int i = i0 + k * (int)blockDim.x;
      if (i < n) v[k] = *src(i);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int i = i0 + k * (int)blockDim.x;
      if (i < n) {
        int pl;
        raw[dst(i, pl)] = v[k];
        if (pl != cur) {
          if (cur >= 0) atomicMax(&in[cur], m);
          cur = pl;
          m = 0;
        }
        m = fx_max(m, v[k]);
      }
    }
  }
  if (cur >= 0) atomicMax(&in[cur], m);
}

// After the largest components are known (behind a __syncthreads): the words of
// the planes and, where one is out of the ordinary, its scaling in the tile.
// Returns whether any is; ends with a __syncthreads.
template <typename DST>
__device__ __forceinline__ bool fx_prepare(I2* tile, int n, int nplanes, uint32_t* in, DST dst) {
  bool odd = false;
  if ((int)threadIdx.x < nplanes) {
    const uint32_t code = fx_classify(in[threadIdx.x]);
    odd = (code >> 16) != 0u;
    in[threadIdx.x] = code;
  }
  odd = __syncthreads_or(odd);
  if (odd) {
    double2* raw = reinterpret_cast<double2*>(tile);
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      int pl;
      double2& v = raw[dst(i, pl)];
      const uint32_t k = in[pl] >> 16;
      if (k == FX_NONFINITE) v = make_double2(0.0, 0.0);
      else if (k != 0u) v = make_double2(scalbn(v.x, k == FX_UP ? FX_ODD_SCALE : -FX_ODD_SCALE),
                                         scalbn(v.y, k == FX_UP ? FX_ODD_SCALE : -FX_ODD_SCALE));
    }
    __syncthreads();
  }
  return odd;
}

template <int SIGN>
__global__ void __launch_bounds__(FX_MAX_THREADS, 2) fft_xy_fx_kernel(Geom g, const __grid_constant__ FxPass P,
                                                        double2* __restrict__ data, const int4* __restrict__ twg,
                                                        const short* __restrict__ posg, int fpb, CopyDiv cd, Batch B) {
  if (batch_skip(B)) return;
  data += blockIdx.z * B.s_delta;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int Lx = g.L[0], Ly = g.L[1];
  int4* tw;
  short* pos;
  FxPlanes* ps;
  I2* tile = fx_setup(smem_raw, twg, posg, Lx, Ly, &tw, &pos, &ps);
  const int RS = Lx + 1, PS = Ly * RS;
  const int plane = Lx * Ly;
  double2* fld = data + (int64_t)(blockIdx.y * fpb) * g.V + (int64_t)blockIdx.x * plane;
  __syncthreads();
  const int n = fpb * plane;
  auto dst = [&](int i, int& pl) {
    const int f = (int)cd.a.div((uint32_t)i), r = i - f * plane, y = (int)cd.b.div((uint32_t)r), x = r - y * Lx;
    pl = f;
    return f * PS + pos[Lx + y] * RS + pos[x];
  };
  fx_load(
      tile, n, ps->t[0].in,
      [&](int i) {
        const int f = (int)cd.a.div((uint32_t)i);
        return &fld[(int64_t)f * g.V + (i - f * plane)];
      },
      dst);
  __syncthreads();
  const bool odd = fx_prepare(tile, n, fpb, ps->t[0].in, dst);
  fx_plane<SIGN, true, true>(tile, P, P.p[0], tw, fpb, &ps->t[0]);
  auto out = [&](auto convert) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const int f = (int)cd.a.div((uint32_t)i), r = i - f * plane, y = (int)cd.b.div((uint32_t)r), x = r - y * Lx;
      fld[(int64_t)f * g.V + r] = convert(tile[f * PS + y * RS + x], ps->t[0].in[f]);
    }
  };
  if (!odd) out(FxOut());
  else out(FxOutAny());
}

// MODE as launch_fft_zt: 0 forward, filter, inverse; -1 / +1 one transform.
template <int MODE, bool LRN>
__global__ void __launch_bounds__(FX_MAX_THREADS, 2)
fft_zt_filter_fx_kernel(Geom g, const __grid_constant__ FxPass P, double2* __restrict__ data,
                        const int4* __restrict__ twg, const short* __restrict__ posg, const double* __restrict__ K,
                        int xc, LearnedIO lio, int4 H, CopyDiv cd, Batch B) {
  if (batch_skip(B)) return;
  data += blockIdx.z * B.s_delta;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int Lx = g.L[0], Ly = g.L[1], Lz = g.L[2], Lt = g.L[3];
  int4* tw;
  short* pos;
  FxPlanes* ps;
  I2* tile = fx_setup(smem_raw, twg + Lx + Ly, posg + Lx + Ly, Lz, Lt, &tw, &pos, &ps);
  const int TS = Lz * xc + 1;
  const int nxb = Lx / xc;
  const int x0 = (blockIdx.x % nxb) * xc, y = blockIdx.x / nxb;
  double2* fld = data + (int64_t)blockIdx.y * g.V;
  const int n = Lz * Lt * xc;
  const int64_t sxy = (int64_t)y * Lx + x0;
  const int64_t plane = (int64_t)Lx * Ly;
  __syncthreads();
#define LGF_ZT_IDX(i)                                                       \
  const int zt = (int)cd.a.div((uint32_t)(i)), xi = (i) - zt * xc;          \
  const int t = (int)cd.b.div((uint32_t)zt), z = zt - t * Lz;
  auto dst = [&](int i, int& pl) {
    LGF_ZT_IDX(i)
    pl = xi;
    return pos[Lz + t] * TS + pos[z] * xc + xi;
  };
  fx_load(
      tile, n, ps->t[0].in,
      [&](int i) {
        const int zt = (int)cd.a.div((uint32_t)i);
        return &fld[(int64_t)zt * plane + sxy + (i - zt * xc)];
      },
      dst);
  __syncthreads();
  bool odd = fx_prepare(tile, n, xc, ps->t[0].in, dst);
  fx_plane<(MODE > 0 ? +1 : -1), true, false>(tile, P, P.p[0], tw, xc, &ps->t[0]);
  if (MODE != 0) {
    auto out = [&](auto convert) {
      for (int i = threadIdx.x; i < n; i += blockDim.x) {
        LGF_ZT_IDX(i)
        fld[(int64_t)zt * plane + sxy + xi] = convert(tile[t * TS + z * xc + xi], ps->t[0].in[xi]);
      }
    };
    if (!odd) out(FxOut());
    else out(FxOutAny());
    return;
  }
  // the filter in FP64, back into the tile; xc divides the CTA size, so a
  // thread stays in one x column
  const int col = (int)threadIdx.x % xc;
  auto filter = [&](auto convert) {
    const int kit = LRN ? lio.st->iter : 0;
    const bool learned = LRN && lio.mtab != nullptr && lio.st->use_m != 0;
    const float* mtab = lio.mtab + (int64_t)(kit & 1) * lio.nclass;
    uint32_t* snap = (LRN && lio.snap != nullptr) ? lio.snap + ((int64_t)(kit & 1) * 4 + blockIdx.y) * g.V : nullptr;
    const int fy = min(y, Ly - y);
    const uint32_t word = ps->t[0].in[col];
    uint32_t m = 0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      LGF_ZT_IDX(i)
      double k = __ldg(&K[(int64_t)zt * plane + sxy + xi]);
      if (learned) {
        const int kx = x0 + xi;
        const int fx = min(kx, Lx - kx), fz = min(z, Lz - z), ft = min(t, Lt - t);
        k *= (double)__ldg(&mtab[((ft * H.z + fz) * H.y + fy) * H.x + fx]);
      }
      double2* e = reinterpret_cast<double2*>(&tile[t * TS + z * xc + xi]);
      const double2 v = convert(*reinterpret_cast<const I2*>(e), word);
      if (LRN && snap != nullptr) snap[(int64_t)zt * plane + sxy + xi] = bf16x2_of<double>(v);
      const double2 w = make_double2(v.x * k, v.y * k);
      m = fx_max(m, w);
      *e = w;
    }
    atomicMax(&ps->t[1].in[col], m);
  };
  if (!odd) filter(FxOut());
  else filter(FxOutAny());
  __syncthreads();
  odd = fx_prepare(tile, n, xc, ps->t[1].in, [&](int i, int& pl) {
    LGF_ZT_IDX(i)
    pl = xi;
    return t * TS + z * xc + xi;
  });
  fx_plane<+1, false, false>(tile, P, P.p[1], tw, xc, &ps->t[1]);
  auto out = [&](auto convert) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      LGF_ZT_IDX(i)
      fld[(int64_t)zt * plane + sxy + xi] =
          convert(tile[pos[Lz + t] * TS + pos[z] * xc + xi], ps->t[1].in[xi]);
    }
  };
  if (!odd) out(FxOut());
  else out(FxOutAny());
#undef LGF_ZT_IDX
}

template <bool EXPG>
__global__ void __launch_bounds__(FX_C_THREADS)
fft_xy_inv_gauge_fx_kernel(Geom g, const __grid_constant__ FxPass P, const double2* __restrict__ data,
                           const int4* __restrict__ twg, const short* __restrict__ posg, double2* __restrict__ gf,
                           double2* __restrict__ Gf, const DevState* __restrict__ st, CopyDiv cd, Batch B) {
  if (batch_skip(B)) return;
  const bool near_id = near_identity(st, B);
  data += blockIdx.z * B.s_delta;
  gf += blockIdx.z * B.s_g;
  if (Gf != nullptr) Gf += blockIdx.z * B.s_G;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int Lx = g.L[0], Ly = g.L[1];
  int4* tw;
  short* pos;
  FxPlanes* ps;
  I2* tile = fx_setup(smem_raw, twg, posg, Lx, Ly, &tw, &pos, &ps);
  const int RS = Lx + 1, PS = Ly * RS;
  const int plane = Lx * Ly;
  const double2* fld = data + (int64_t)blockIdx.x * plane;
  __syncthreads();
  auto dst = [&](int i, int& pl) {
    const int f = (int)cd.a.div((uint32_t)i), r = i - f * plane, y = (int)cd.b.div((uint32_t)r), x = r - y * Lx;
    pl = f;
    return f * PS + y * RS + x;
  };
  fx_load(
      tile, 4 * plane, ps->t[0].in,
      [&](int i) {
        const int f = (int)cd.a.div((uint32_t)i);
        return &fld[(int64_t)f * g.V + (i - f * plane)];
      },
      dst);
  __syncthreads();
  fx_prepare(tile, 4 * plane, 4, ps->t[0].in, dst);
  fx_plane<+1, false, true>(tile, P, P.p[0], tw, 4, &ps->t[0]);
  for (int i = threadIdx.x; i < plane; i += blockDim.x) {
    const int y = (int)cd.b.div((uint32_t)i), x = i - y * Lx;
    const int o = pos[Lx + y] * RS + pos[x];
    const int64_t s = (int64_t)blockIdx.x * plane + i;
    if (!EXPG && !near_id) {
      int64_t A[8];
      bool ok = true;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const I2 v = tile[k * PS + o];
        const int ex = fx_true_exp(ps->t[0].in[k]);
        A[2 * k] = fx_unit58(v.x, ex, ok);
        A[2 * k + 1] = fx_unit58(v.y, ex, ok);
      }
      if (ok) {
        gauge_site_fx(A, g.V, s, gf, Gf);
        continue;
      }
    }
    double2 f[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) f[k] = fx_out_any(tile[k * PS + o], ps->t[0].in[k]);
    gauge_site_fp64<EXPG>(f[0], f[1], f[2], f[3], g.V, s, gf, Gf, near_id);
  }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------

void fft_twiddles(const int L[4], bool fixed, std::vector<double2>& tw) {
  const int nt = L[0] + L[1] + L[2] + L[3];
  tw.resize((size_t)(fixed ? 2 * nt : nt));
  int off = 0;
  for (int mu = 0; mu < 4; ++mu) {
    for (int m = 0; m < L[mu]; ++m) {
      const double a = -2.0 * M_PI * (double)m / (double)L[mu];
      tw[off + m] = make_double2(std::cos(a), std::sin(a));
    }
    if (fixed) fixed_roots(L[mu], reinterpret_cast<int*>(tw.data() + nt + off));
    off += L[mu];
  }
}

static const int4* fx_table(const Geom& g, const double2* tw) {
  return reinterpret_cast<const int4*>(tw + g.L[0] + g.L[1] + g.L[2] + g.L[3]);
}

// The (x, y) planes of nf fields side by side in a tile.
static FxPass xy_pass(const FFTPlan& p, int Lx, int Ly, int nf, bool dit) {
  const int RS = Lx + 1, PS = Ly * RS;
  return FxPass{{p.d[0], p.d[1]},
                {make_lines(nf * Ly, Ly, RS, PS, 1), make_lines(nf * Lx, Lx, 1, PS, RS)},
                {fx_program(p.d, 0, dit), FxProgram{}}};
}

template <typename K, typename... Args>
static cudaError_t fx_launch(K kernel, dim3 grid, int threads, size_t smem, cudaStream_t s, const Args&... args) {
  const cudaError_t e = allow_smem(kernel, smem);
  if (e != cudaSuccess) return e;
  kernel<<<grid, threads, smem, s>>>(args...);
  return cudaGetLastError();
}

cudaError_t launch_fft_xy_fx(const Geom& g, const FFTPlan& p, double2* data, const double2* tw, const short* pos,
                             int sign, int nfields, cudaStream_t s, const Batch& B) {
  int fpb = std::min(p.fpb_xy, nfields);
  while (nfields % fpb) fpb /= 2;
  const int Lx = g.L[0], Ly = g.L[1];
  const size_t smem = plane_header_bytes(Lx, Ly, 8) + (size_t)fpb * Ly * (Lx + 1) * sizeof(double2);
  const dim3 grid((unsigned)(g.L[2] * g.L[3]), (unsigned)(nfields / fpb), (unsigned)B.n);
  const FxPass P = xy_pass(p, Lx, Ly, fpb, true);
  const CopyDiv cd{FastDiv::make((uint32_t)(Lx * Ly)), FastDiv::make((uint32_t)Lx)};
  return fx_launch(sign < 0 ? fft_xy_fx_kernel<-1> : fft_xy_fx_kernel<+1>, grid, p.threads_xy, smem, s, g, P, data,
                   fx_table(g, tw), pos, fpb, cd, B);
}

cudaError_t launch_fft_zt_fx(const Geom& g, const FFTPlan& p, double2* data, const double2* tw, const short* pos,
                             const double* K, int mode, int nfields, cudaStream_t s, const LearnedIO& lio,
                             const Batch& B) {
  const dim3 grid((unsigned)(g.L[0] / p.xc * g.L[1]), (unsigned)nfields, (unsigned)B.n);
  const bool lrn = mode == 0 && (lio.mtab != nullptr || lio.snap != nullptr);
  const int4 H = make_int4(g.L[0] / 2 + 1, g.L[1] / 2 + 1, g.L[2] / 2 + 1, g.L[3] / 2 + 1);
  const int xc = p.xc, Lz = g.L[2], Lt = g.L[3], TS = Lz * xc + 1;
  const FxPass P{{p.d[2], p.d[3]},
                 {make_lines(Lt * xc, xc, 1, TS, xc), make_lines(Lz * xc, xc, 1, xc, TS)},
                 {fx_program(p.d + 2, 0, true), fx_program(p.d + 2, 1, false)}};
  const CopyDiv cd{FastDiv::make((uint32_t)xc), FastDiv::make((uint32_t)Lz)};
  auto kernel = mode < 0   ? fft_zt_filter_fx_kernel<-1, false>
                : mode > 0 ? fft_zt_filter_fx_kernel<+1, false>
                : lrn      ? fft_zt_filter_fx_kernel<0, true>
                           : fft_zt_filter_fx_kernel<0, false>;
  return fx_launch(kernel, grid, p.threads_zt, p.smem_zt, s, g, P, data, fx_table(g, tw), pos, K, xc, lio, H, cd, B);
}

cudaError_t launch_xy_inv_gauge_fx(const Geom& g, const FFTPlan& p, const double2* data, const double2* tw,
                                   const short* pos, double2* gfield, double2* Gfield, const DevState* st,
                                   cudaStream_t s, const Batch& B, bool exact_exp) {
  const int Lx = g.L[0], Ly = g.L[1];
  const FxPass P = xy_pass(p, Lx, Ly, 4, false);
  const CopyDiv cd{FastDiv::make((uint32_t)(Lx * Ly)), FastDiv::make((uint32_t)Lx)};
  const dim3 grid((unsigned)(g.L[2] * g.L[3]), 1, (unsigned)B.n);
  return fx_launch(exact_exp ? fft_xy_inv_gauge_fx_kernel<true> : fft_xy_inv_gauge_fx_kernel<false>, grid, p.threads_c,
                   p.smem_c, s, g, P, data, fx_table(g, tw), pos, gfield, Gfield, st, cd, B);
}

}  // namespace lgf
