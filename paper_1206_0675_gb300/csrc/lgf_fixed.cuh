// Fixed-point arithmetic for FP64 data whose values are bounded by one
// (elements of SU(3) matrices), on the integer pipe.
//
// Why: a GB300 SM issues 2 FP64 operations per clock but 64 IMAD.WIDE
// (32 x 32 + 64 -> 64 bits), so a real multiply-add of two 60-bit fixed-point
// numbers, three IMAD.WIDE, takes 3/64 clock against 1/2 clock of the FP64 pipe.
// Its rounding is finer too: every product is kept to 2^-60 absolute, while
// an FP64 operation on numbers of order one rounds at 2^-54 (measured on the
// link update of random SU(3) fields: see update_kernel).
//
// Format: a = (H 2^30 + L) 2^-60 with |a| < FX_LIM = 1.125; H and L are
// 32-bit signed words, |H| <= 1.125 2^30 and |L| <= 2^29 (centred, so that what
// is dropped has no preferred sign: a bias of a few 2^-62 per product adds up
// over the steps of a converging field, whose theta it shows in).  An
// accumulator keeps two 64-bit sums, hi += H H' (unit 2^-60) and mid += H L' +
// L H' (unit 2^-90); L L' < 2^-62 is dropped.  Six real products (one
// component of a row times column) stay below 6 (1.125 2^30)^2 < 2^63 in hi
// and 12 (1.125 2^30) 2^29 < 2^63 in mid, so sums never overflow whatever the
// matrices are, as long as each entry is below FX_LIM.  Callers test that
// (fx_bad) and take an FP64 path otherwise, which also carries infinities
// and NaN through.
#pragma once

#include "lgf_common.cuh"

namespace lgf {

// high word of 1.125
constexpr uint32_t FX_LIM_HI = 0x3ff20000u;
// Links near the identity: FP64 rounds small entries finer than the fixed-point
// unit, so theta of a converged field of links 1 + O(eps) falls with eps^2 in
// FP64, and levels off in fixed point.  Where all off-diagonal entries of a link
// (01, 02, 12) are below these, its warp takes FP64 as a whole (a warp would do
// both otherwise), decided before any arithmetic.
// High word of 2^-5: in the measurement and the hits, whose sums of links have
// the unit 2^-58 or 2^-59.  theta of 8^4 levels off (fixed point / FP64) at
// 1.7e-33 / 1.4e-33 for eps = 0.06, of whose warps 98 % are below the line, and at
// 1.1e-33 / 5.4e-33 for 0.12, of whose warps 12 % are; 0.1 % are for eps = 0.3.
constexpr uint32_t FX_NEAR_HI = 0x3fa00000u;
// High word of 2^-7: in the products of single links, unit 2^-60.
constexpr uint32_t FX_WEAK_HI = 0x3f800000u;

// c + a b with a 64-bit sum: one IMAD.WIDE.  (Both factors have to look like
// signed 32-bit words to the compiler, which turns products with a factor of
// known range or sign into 64 x 64 bit ones and differences: every operand
// passes through fx_opaque.  Written in PTX the sum costs a register move per
// product.)
__device__ __forceinline__ int64_t mad_wide(int a, int b, int64_t c) { return c + (int64_t)a * b; }
__device__ __forceinline__ int fx_opaque(int a) {
  asm("" : "+r"(a));
  return a;
}

struct Fx {
  int h, l;
};
struct FxC {
  Fx x, y;
};

// Accumulates max |a| (as high words) so that one comparison tests many
// entries: bad if the result is >= FX_LIM_HI (infinities and NaN included).
__device__ __forceinline__ uint32_t fx_max(uint32_t m, double a) {
  return max(m, (uint32_t)__double2hiint(a) & 0x7fffffffu);
}
__device__ __forceinline__ uint32_t fx_max(uint32_t m, double2 a) { return fx_max(fx_max(m, a.x), a.y); }

// x >> s for 0 <= s, zero from s = 64 on (PTX shifts clamp their count).
__device__ __forceinline__ uint64_t shr64_clamp(uint64_t x, uint32_t s) {
  uint64_t r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
  return r;
}
__device__ __forceinline__ uint32_t shr32_clamp(uint32_t x, uint32_t s) {
  uint32_t r;
  asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(s));
  return r;
}

// The operand of a number in units of 2^-60.
__device__ __forceinline__ Fx fx_operand(int64_t r60) {
  return Fx{fx_opaque((int)((r60 + ((int64_t)1 << 29)) >> 30)), fx_opaque((int)((uint32_t)r60 << 2) >> 2)};
}

// Fixed point from FP64 in units of 2^-60, |a| < 2; what lies below is cut off.
// With the leading one at bit 63 the significand M has the value
// M 2^(e - 1086), so the magnitude in units of 2^-60 is M >> (1026 - e).
__device__ __forceinline__ int64_t fx60_from(double a) {
  const uint32_t hi = (uint32_t)__double2hiint(a), lo = (uint32_t)__double2loint(a);
  const uint32_t mh = __funnelshift_l(lo, hi, 11) | 0x80000000u, ml = lo << 11;
  const int64_t sg = (int64_t)((int)hi >> 31);
  return ((int64_t)shr64_clamp(((uint64_t)mh << 32) | ml, 1026u - ((hi >> 20) & 0x7ffu)) ^ sg) - sg;
}
__device__ __forceinline__ Fx fx_from(double a) { return fx_operand(fx60_from(a)); }
__device__ __forceinline__ FxC fx_from(double2 a) { return FxC{fx_from(a.x), fx_from(a.y)}; }
__device__ __forceinline__ Fx fx_neg(Fx a) { return Fx{fx_opaque(-a.h), fx_opaque(-a.l)}; }
__device__ __forceinline__ FxC fx_neg(FxC a) { return FxC{fx_neg(a.x), fx_neg(a.y)}; }
__device__ __forceinline__ FxC fx_conj(FxC a) { return FxC{a.x, fx_neg(a.y)}; }

// Two-part accumulator of real products.
struct FxAcc {
  int64_t hi, mid;
};
__device__ __forceinline__ FxAcc fx_zero() { return FxAcc{0, (int64_t)1 << 29}; }  // rounds when mid is shifted by 30
__device__ __forceinline__ void fx_mac(FxAcc& s, Fx a, Fx b) {
  s.hi = mad_wide(a.h, b.h, s.hi);
  s.mid = mad_wide(a.h, b.l, s.mid);
  s.mid = mad_wide(a.l, b.h, s.mid);
}
// s += a b and s += a conj(b) for complex numbers; na = -a where a sign is needed
__device__ __forceinline__ void fx_cmac(FxAcc& re, FxAcc& im, const FxC& a, Fx nay, const FxC& b) {
  fx_mac(re, a.x, b.x);
  fx_mac(re, nay, b.y);
  fx_mac(im, a.x, b.y);
  fx_mac(im, a.y, b.x);
}
__device__ __forceinline__ void fx_cmacc(FxAcc& re, FxAcc& im, const FxC& a, Fx nax, const FxC& b) {
  fx_mac(re, a.x, b.x);
  fx_mac(re, a.y, b.y);
  fx_mac(im, a.y, b.x);
  fx_mac(im, nax, b.y);
}

// Twice and four times a sum, rounded to 2^-60 after the multiplication.
__device__ __forceinline__ FxAcc fx_zero_x2() { return FxAcc{0, (int64_t)1 << 28}; }
__device__ __forceinline__ int64_t fx_sum60_x2(const FxAcc& s) { return 2 * s.hi + (s.mid >> 29); }
__device__ __forceinline__ FxAcc fx_zero_x4() { return FxAcc{0, (int64_t)1 << 27}; }
__device__ __forceinline__ int64_t fx_sum60_x4(const FxAcc& s) { return 4 * s.hi + (s.mid >> 28); }

// An accumulated sum r in units of 2^-60, and its test against FX_LIM: sums
// over rows and columns of matrices that are far from unitary can exceed it
// although every entry passed fx_max.  t collects the largest r + FX_LIM;
// bad if it reaches 2 FX_LIM.
constexpr uint32_t FX_SUM_OFF = 0x12000000u;  // 1.125 in units of 2^-28
__device__ __forceinline__ int64_t fx_sum60(const FxAcc& s, uint32_t& t) {
  const int64_t r = s.hi + (s.mid >> 30);
  t = max(t, (uint32_t)(r >> 32) + FX_SUM_OFF);
  return r;
}
__device__ __forceinline__ bool fx_bad(uint32_t m, uint32_t t) { return m >= FX_LIM_HI || t >= 2u * FX_SUM_OFF; }
// 64-bit fixed point in units of 2^-K from FP64, |a| < 2 (zero for what lies
// below): 2^-58 for sums of up to 16 entries, 2^-59 for sums of up to 8.
template <int K> __device__ __forceinline__ int64_t fxk_from(double a) {
  const uint32_t hi = (uint32_t)__double2hiint(a), lo = (uint32_t)__double2loint(a);
  const uint32_t mh = __funnelshift_l(lo, hi, 11) | 0x80000000u, ml = lo << 11;
  const uint32_t s = 1086u - K - ((hi >> 20) & 0x7ffu);
  const int64_t sg = (int64_t)((int)hi >> 31);
  return ((int64_t)shr64_clamp(((uint64_t)mh << 32) | ml, s) ^ sg) - sg;
}
__device__ __forceinline__ int64_t fx58_from(double a) { return fxk_from<58>(a); }
__device__ __forceinline__ Fx fx_operand58(int64_t a58) { return fx_operand(a58 << 2); }

// FP64 value of a 64-bit integer n times 2^-K, rounded to nearest, on the
// FP64 pipe: the two halves are placed into the significands of doubles of
// fixed exponent, whose offsets the two additions take away (the first is
// exact).
template <int K> __device__ __forceinline__ double fx_to_double_fp(int64_t n) {
  const double h = __hiloint2double(0x45300000 - (K << 20), (int)((uint32_t)(n >> 32) ^ 0x80000000u));
  const double l = __hiloint2double(0x43300000 - (K << 20), (int)(uint32_t)n);
  // 2^84 + 2^63 + 2^52, times 2^-K
  const double off = __hiloint2double(0x45300000 - (K << 20), (int)0x80100000u);
  return (h - off) + l;
}

// The same on the integer pipe, for |n| >= 2^32 (ok = false below): leading
// one to bit 62, rounding of the 10 bits below the significand, ties to even,
// then the significand's leading one and a carry add into the exponent.
template <int K> __device__ __forceinline__ double fx_to_double_int(int64_t n, bool& ok) {
  const int sg = (int)(n >> 63);
  const uint64_t u = (uint64_t)((n ^ (int64_t)sg) - (int64_t)sg);
  const uint32_t uh = (uint32_t)(u >> 32);
  ok = ok && uh != 0u;
  const int lz = __clz((int)uh);
  const uint64_t v = u << (lz - 1);
  const uint64_t m = (v + 0x1ffull + (((uint32_t)v >> 10) & 1u)) >> 10;
  const uint32_t ew = (uint32_t)(1023 + 62 - K) * 0x100000u - (uint32_t)lz * 0x100000u;
  const uint32_t rh = (uint32_t)(m >> 32) + ew;
  return __hiloint2double((int)(rh | ((uint32_t)sg & 0x80000000u)), (int)(uint32_t)m);
}

// Entry (k l) of the third row of an SU(3) matrix from its first two rows:
// conj(a_k b_l - a_l b_k), real part and imaginary part.
__device__ __forceinline__ void fx_cross_conj(FxAcc& re, FxAcc& im, const FxC& ak, const FxC& al, const FxC& bk,
                                              const FxC& bl) {
  const Fx nakx = fx_neg(ak.x), naky = fx_neg(ak.y), nalx = fx_neg(al.x);
  fx_mac(re, ak.x, bl.x);
  fx_mac(re, naky, bl.y);
  fx_mac(re, nalx, bk.x);
  fx_mac(re, al.y, bk.y);
  fx_mac(im, nakx, bl.y);
  fx_mac(im, naky, bl.x);
  fx_mac(im, al.x, bk.y);
  fx_mac(im, al.y, bk.x);
}

// ---------------------------------------------------------------------------
// block floating point: 64-bit integers with a common exponent per block
// ---------------------------------------------------------------------------

// Integer of an FP64 number in units that make the block's largest magnitude
// fit (see the transform passes): M >> (base - e), rounded, M with its leading
// one at bit 63.  base > 64, so zeros and numbers 2^-64 below the block's
// largest give zero.
__device__ __forceinline__ int64_t bfp_from(double a, uint32_t base) {
  const uint32_t hi = (uint32_t)__double2hiint(a), lo = (uint32_t)__double2loint(a);
  const uint32_t mh = __funnelshift_l(lo, hi, 11) | 0x80000000u, ml = lo << 11;
  const int64_t sg = (int64_t)((int)hi >> 31);
  return ((int64_t)((shr64_clamp(((uint64_t)mh << 32) | ml, base - 1u - ((hi >> 20) & 0x7ffu)) + 1u) >> 1) ^ sg) - sg;
}

// FP64 value of n 2^ex rounded to nearest, where the result is far from the
// ends of the FP64 range or zero.
__device__ __forceinline__ double bfp_to_double(int64_t n, int ex) {
  const int sg = (int)(n >> 63);
  const uint64_t u = (uint64_t)((n ^ (int64_t)sg) - (int64_t)sg);
  const uint32_t uh = (uint32_t)(u >> 32);
  if (uh == 0u) {  // rare: zeros and numbers 2^-29 below the block's largest
    const double r = fx_to_double_fp<0>(n);
    return r == 0.0 ? r : __hiloint2double(__double2hiint(r) + ex * 0x100000, __double2loint(r));
  }
  const int lz = __clz((int)uh);
  const uint64_t m = ((u << (lz - 1)) + 0x200ull) >> 10;
  const uint32_t rh = (uint32_t)(m >> 32) + (uint32_t)(1023 + 62 + ex - lz) * 0x100000u;
  return __hiloint2double((int)(rh | ((uint32_t)sg & 0x80000000u)), (int)(uint32_t)m);
}

// X (|X| < 2^61) as two limbs, X = h 2^30 + l.
struct Bfp2 {
  int h, l;
};
__device__ __forceinline__ Bfp2 bfp_limbs(int64_t x) {
  return Bfp2{fx_opaque((int)(x >> 30)), fx_opaque((int)((uint32_t)x & 0x3fffffffu))};
}

// Real and complex products with a constant or a root of unity w, |w| <= 1,
// w = h 2^-30 + l 2^-60 (|l| <= 2^29): three multiply-adds per real product,
// rounded to the nearest unit.  Of l l' 2^-60, up to half a unit, the mean over
// the low limbs l of x, l' 2^-31, goes in with the rounding: dropped, it adds the
// same to every product with one root, and a line of 81 (four stages with
// sqrt(3)/2) gathered 30 times the error of one of 64 in its low modes.
__device__ __forceinline__ int64_t bfp_mul(int64_t x, int wh, int wl) {
  const Bfp2 a = bfp_limbs(x);
  const int64_t mid = mad_wide(a.l, wh, mad_wide(a.h, wl, ((int64_t)1 << 29) + (wl >> 1)));
  return mad_wide(a.h, wh, mid >> 30);
}

// ---------------------------------------------------------------------------
// g of FP64 lanes, stored as fixed-point operands
// ---------------------------------------------------------------------------

// One complex entry is 16 bytes, and the nine entries of a site have one of two
// forms.  Operands: four words (re h, re l, im h, im l), so that the update reads
// them as they are (five threads read every g(x): converting FP64 entries cost
// the update a seventh of its instructions).  FP64 numbers (re, im): where the
// field is near the identity (DevState::near_id) -- g - 1 is then small and the
// unit 2^-60 is far above what FP64 keeps of it -- and where g is not finite.
// The forms are told apart by the second word of the first entry: l of an
// operand lies in [-2^29, 2^29), the high word of an FP64 number does not
// unless its magnitude is below 2^-511 (of a positive one) or from 2^513 (of a
// negative one), which the store replaces.
__device__ __forceinline__ bool fxg_is_fp64(int4 first) {
  return (uint32_t)first.y + 0x20000000u >= 0x40000000u;
}
__device__ __forceinline__ FxC fxg_unpack(int4 w) { return FxC{Fx{w.x, w.y}, Fx{w.z, w.w}}; }
__device__ __forceinline__ int4 fxg_pack(const FxC& a) { return make_int4(a.x.h, a.x.l, a.y.h, a.y.l); }
__device__ __forceinline__ double2 fxg_fp64(int4 w) {
  return make_double2(__hiloint2double(w.y, w.x), __hiloint2double(w.w, w.z));
}
__device__ __forceinline__ int4 fxg_of_fp64(double2 v) {
  return make_int4(__double2loint(v.x), __double2hiint(v.x), __double2loint(v.y), __double2hiint(v.y));
}
__device__ __forceinline__ double fx_value(Fx a) { return fx_to_double_fp<60>(((int64_t)a.h << 30) + a.l); }

// g in FP64 from its entries p[e stride].
__device__ __forceinline__ void fxg_load(const int4* p, int64_t stride, M3<double>& M) {
  if (fxg_is_fp64(p[0])) {
#pragma unroll
    for (int e = 0; e < 9; ++e) M.e[e / 3][e % 3] = fxg_fp64(p[e * stride]);
  } else {
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      const FxC w = fxg_unpack(p[e * stride]);
      M.e[e / 3][e % 3] = make_double2(fx_value(w.x), fx_value(w.y));
    }
  }
}
__device__ __forceinline__ void fxg_load(const double2* gf, int64_t V, int64_t s, M3<double>& M) {
  fxg_load(reinterpret_cast<const int4*>(gf) + s, V, M);
}
// The stores, from FP64 rows: as FP64 numbers, and as operands (NaN in all
// entries where one is outside their range).
__device__ __forceinline__ void fxg_store_fp64(double2* __restrict__ gf, int64_t V, int64_t s, const double2 a[3],
                                               const double2 b[3], const double2 c[3]) {
  int4* p = reinterpret_cast<int4*>(gf);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    int4 w = fxg_of_fp64(a[j]);
    if (j == 0 && !fxg_is_fp64(w)) {
      w.y = w.y >= 0 ? 0x20b00000 : 0x7ff80000;  // 2^-500 for 0, NaN for what is not finite
      w.x = 0;
    }
    p[j * V + s] = w;
    p[(3 + j) * V + s] = fxg_of_fp64(b[j]);
    p[(6 + j) * V + s] = fxg_of_fp64(c[j]);
  }
}
__device__ __forceinline__ void fxg_store(double2* __restrict__ gf, int64_t V, int64_t s, const double2 a[3],
                                          const double2 b[3], const double2 c[3]) {
  int4* p = reinterpret_cast<int4*>(gf);
  uint32_t m = 0;
#pragma unroll
  for (int j = 0; j < 3; ++j) m = fx_max(fx_max(fx_max(m, a[j]), b[j]), c[j]);
  const bool bad = m >= FX_LIM_HI;
  const int4 nan = make_int4(0, 0x7ff80000, 0, 0x7ff80000);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    p[j * V + s] = bad ? nan : fxg_pack(fx_from(a[j]));
    p[(3 + j) * V + s] = bad ? nan : fxg_pack(fx_from(b[j]));
    p[(6 + j) * V + s] = bad ? nan : fxg_pack(fx_from(c[j]));
  }
}

// y/2 in units of 2^-60 for y = 1/sqrt(n), n in units of 2^-60 and
// 1/16 <= n < 2: the FP32 estimate, a 24-bit integer, and one third-order step
// (e = 1 - n y0^2 below 2^-19 in magnitude, so 5 e^3 / 16 is below 2^-58 of y0;
// see rsqrt_fp64).
__device__ __forceinline__ int64_t fx_half_rsqrt(int64_t n) {
  const float f = (float)(int)(n >> 30) * 9.3132257e-10f;  // 2^-30
  const int y0 = __float2int_rn(rsqrtf(f) * 4194304.f);    // unit 2^-22
  const int64_t t = ((int64_t)((int)(n >> 30)) * y0 << 8) + ((int64_t)((int)n & 0x3fffffff) * y0 >> 22);
  const int64_t q = ((int64_t)((int)(t >> 30)) * y0 << 8) + ((int64_t)((int)t & 0x3fffffff) * y0 >> 22);
  const int64_t e = ((int64_t)1 << 60) - q;
  const int eh = (int)(e >> 20);
  const int64_t c = (e >> 1) + (3 * ((int64_t)eh * eh) >> 23);
  return ((int64_t)y0 << 37) + ((int64_t)((int)(c >> 20)) * y0 >> 3) + ((int64_t)((int)c & 0xfffff) * y0 >> 23);
}

// ---------------------------------------------------------------------------
// updated links
// ---------------------------------------------------------------------------

// Third row (as operands or sums) from rows that are operands.
__device__ __forceinline__ void fx_third_row(const FxC a[3], const FxC b[3], int64_t c[3][2], uint32_t& t) {
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    FxAcc re = fx_zero(), im = fx_zero();
    fx_cross_conj(re, im, a[(j + 1) % 3], a[(j + 2) % 3], b[(j + 1) % 3], b[(j + 2) % 3]);
    c[j][0] = fx_sum60(re, t);
    c[j][1] = fx_sum60(im, t);
  }
}

// An updated link in FP64 from the sums of its rows 1-2 (n, units of 2^-60)
// and, for 18-real storage, of row 3 (n3).  Row 3 converts on the FP64 pipe,
// which is idle otherwise.
template <int ROWS>
__device__ __forceinline__ void fx_link_to_double(const int64_t n[2][3][2], const int64_t n3[3][2],
                                                  double2 o[ROWS][3]) {
  bool big = true;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      o[i][j] = make_double2(fx_to_double_int<60>(n[i][j][0], big), fx_to_double_int<60>(n[i][j][1], big));
  if (!big) {  // an entry below 2^-28, zeros among them
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j)
        o[i][j] = make_double2(fx_to_double_fp<60>(n[i][j][0]), fx_to_double_fp<60>(n[i][j][1]));
  }
  if (ROWS == 3) {
#pragma unroll
    for (int j = 0; j < 3; ++j) o[2][j] = make_double2(fx_to_double_fp<60>(n3[j][0]), fx_to_double_fp<60>(n3[j][1]));
  }
}

}  // namespace lgf
