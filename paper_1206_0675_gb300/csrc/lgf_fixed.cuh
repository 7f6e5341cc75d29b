// Fixed-point arithmetic for FP64 data whose values are bounded by one
// (elements of SU(3) matrices), on the integer pipe.
//
// Why: a GB300 SM issues 2 FP64 operations per clock but 64 IMAD.WIDE
// (32 x 32 + 64 -> 64 bits), so a real multiply-add of two 59-bit fixed-point
// numbers, three IMAD.WIDE, takes 3/64 clock against 1/2 clock of the FP64 pipe.
// Its rounding is finer too: every product is kept to 2^-60 absolute, while
// an FP64 operation on numbers of order one rounds at 2^-54 (measured on the
// link update of random SU(3) fields: see update_kernel).
//
// Format: a = (H 2^29 + L) 2^-59 with |a| < FX_LIM = 1.125; H and L are
// 32-bit signed words, |H| <= 1.125 2^30 and |L| < 2^29.  An accumulator
// keeps two 64-bit sums, hi += H H' (unit 2^-60) and mid += H L' + L H'
// (unit 2^-89); L L' < 2^-60 is dropped.  Six real products (one component
// of a row times column) stay below 6 (1.125 2^30)^2 < 2^63 in hi and
// 12 (1.125 2^30) 2^29 < 2^63 in mid, so sums never overflow whatever the
// matrices are, as long as each entry is below FX_LIM.  Callers test that
// (fx_bad) and take an FP64 path otherwise, which also carries infinities
// and NaN through.
#pragma once

#include "lgf_common.cuh"

namespace lgf {

// high word of 1.125
constexpr uint32_t FX_LIM_HI = 0x3ff20000u;
// high word of 2^-12: below it an FP64 rounding (2^-65) is finer than the unit
constexpr uint32_t FX_WEAK_HI = 0x3f300000u;

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

// Fixed point from FP64, |a| < FX_LIM; bits below 2^-59 are cut off.
// With the leading one at bit 63 the significand M has the value
// M 2^(e - 1086), so the magnitude in units of 2^-59 is M >> (1027 - e).
__device__ __forceinline__ Fx fx_from(double a) {
  const uint32_t hi = (uint32_t)__double2hiint(a), lo = (uint32_t)__double2loint(a);
  const uint32_t mh = __funnelshift_l(lo, hi, 11) | 0x80000000u, ml = lo << 11;
  const uint32_t s = 1027u - ((hi >> 20) & 0x7ffu);
  const int sg = (int)hi >> 31;
  const uint32_t h = shr32_clamp(mh, s - 3u);
  const uint32_t l = (uint32_t)shr64_clamp(((uint64_t)mh << 32) | ml, s) & 0x1fffffffu;
  return Fx{((int)h ^ sg) - sg, ((int)l ^ sg) - sg};
}
__device__ __forceinline__ FxC fx_from(double2 a) { return FxC{fx_from(a.x), fx_from(a.y)}; }
__device__ __forceinline__ Fx fx_neg(Fx a) { return Fx{-a.h, -a.l}; }

// Two-part accumulator of real products.
struct FxAcc {
  int64_t hi, mid;
};
__device__ __forceinline__ FxAcc fx_zero() { return FxAcc{0, (int64_t)1 << 28}; }  // rounds when mid is shifted by 29
__device__ __forceinline__ void fx_mac(FxAcc& s, Fx a, Fx b) {
  s.hi += (int64_t)a.h * b.h;
  s.mid += (int64_t)a.h * b.l;
  s.mid += (int64_t)a.l * b.h;
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

// An accumulated sum r in units of 2^-60, and its test against FX_LIM: sums
// over rows and columns of matrices that are far from unitary can exceed it
// although every entry passed fx_max.  t collects the largest r + FX_LIM;
// bad if it reaches 2 FX_LIM.
constexpr uint32_t FX_SUM_OFF = 0x12000000u;  // 1.125 in units of 2^-28
__device__ __forceinline__ int64_t fx_sum60(const FxAcc& s, uint32_t& t) {
  const int64_t r = s.hi + (s.mid >> 29);
  t = max(t, (uint32_t)(r >> 32) + FX_SUM_OFF);
  return r;
}
__device__ __forceinline__ bool fx_bad(uint32_t m, uint32_t t) { return m >= FX_LIM_HI || t >= 2u * FX_SUM_OFF; }
// The sum as an operand of the next product.
__device__ __forceinline__ Fx fx_operand(int64_t r60) {
  return Fx{(int)(r60 >> 30), (int)((uint32_t)(r60 >> 1) & 0x1fffffffu)};
}

// 64-bit fixed point in units of 2^-58 from FP64, |a| < 2 (zero for what lies
// below): for sums of up to 16 entries.
__device__ __forceinline__ int64_t fx58_from(double a) {
  const uint32_t hi = (uint32_t)__double2hiint(a), lo = (uint32_t)__double2loint(a);
  const uint32_t mh = __funnelshift_l(lo, hi, 11) | 0x80000000u, ml = lo << 11;
  const uint32_t s = 1028u - ((hi >> 20) & 0x7ffu);
  const int64_t sg = (int64_t)((int)hi >> 31);
  return ((int64_t)shr64_clamp(((uint64_t)mh << 32) | ml, s) ^ sg) - sg;
}
__device__ __forceinline__ Fx fx_operand58(int64_t a58) {
  return Fx{(int)(a58 >> 28), (int)((uint32_t)(a58 << 1) & 0x1fffffffu)};
}

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

// The same on the integer pipe, for |n| >= 2^32 (ok = false below; ties go
// away from zero): leading one to bit 62, half a unit of the last kept bit,
// then the significand's leading one and a carry add into the exponent.
template <int K> __device__ __forceinline__ double fx_to_double_int(int64_t n, bool& ok) {
  const int sg = (int)(n >> 63);
  const uint64_t u = (uint64_t)((n ^ (int64_t)sg) - (int64_t)sg);
  const uint32_t uh = (uint32_t)(u >> 32);
  ok = ok && uh != 0u;
  const int lz = __clz((int)uh);
  const uint64_t m = ((u << (lz - 1)) + 0x200ull) >> 10;
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
// fit (see the transform passes): M >> (base - e), M with its leading one at
// bit 63.  base >= 100, so zeros and numbers 2^-64 below the block's largest
// give zero.
__device__ __forceinline__ int64_t bfp_from(double a, uint32_t base) {
  const uint32_t hi = (uint32_t)__double2hiint(a), lo = (uint32_t)__double2loint(a);
  const uint32_t mh = __funnelshift_l(lo, hi, 11) | 0x80000000u, ml = lo << 11;
  const int64_t sg = (int64_t)((int)hi >> 31);
  return ((int64_t)shr64_clamp(((uint64_t)mh << 32) | ml, base - ((hi >> 20) & 0x7ffu)) ^ sg) - sg;
}

// FP64 value of n 2^ex rounded to nearest, any n and ex.
static __device__ __noinline__ double bfp_to_double_any(int64_t n, int ex) { return scalbn(fx_to_double_fp<0>(n), ex); }

// The same on the integer pipe where the block's exponents are far from the
// ends of the FP64 range (safe) and |n| >= 2^32.
__device__ __forceinline__ double bfp_to_double(int64_t n, int ex, bool safe) {
  const int sg = (int)(n >> 63);
  const uint64_t u = (uint64_t)((n ^ (int64_t)sg) - (int64_t)sg);
  const uint32_t uh = (uint32_t)(u >> 32);
  if (!safe || uh == 0u) return bfp_to_double_any(n, ex);
  const int lz = __clz((int)uh);
  const uint64_t m = ((u << (lz - 1)) + 0x200ull) >> 10;
  const uint32_t rh = (uint32_t)(m >> 32) + (uint32_t)(1023 + 62 + ex - lz) * 0x100000u;
  return __hiloint2double((int)(rh | ((uint32_t)sg & 0x80000000u)), (int)(uint32_t)m);
}

// X (|X| < 2^61) as two limbs, X = h 2^30 + l.
struct Bfp2 {
  int h, l;
};
__device__ __forceinline__ Bfp2 bfp_limbs(int64_t x) { return Bfp2{(int)(x >> 30), (int)((uint32_t)x & 0x3fffffffu)}; }

// Real and complex products with a constant or a root of unity w, |w| <= 1,
// w = h 2^-30 + l 2^-60 (|l| <= 2^29): three multiply-adds per real product,
// rounded to the nearest unit (l l' 2^-60 is dropped, below 2^-30 of a unit).
__device__ __forceinline__ int64_t bfp_mul(int64_t x, int wh, int wl) {
  const Bfp2 a = bfp_limbs(x);
  int64_t mid = (int64_t)1 << 29;
  mid += (int64_t)a.h * wl;
  mid += (int64_t)a.l * wh;
  return (int64_t)a.h * wh + (mid >> 30);
}

}  // namespace lgf
