// g(x) of one site from its packed filtered divergence: the first-order form
// and the exact exponential, and the store of g (and G <- g G).
#pragma once

#include "lgf_fixed.cuh"
#include "lgf_internal.h"

namespace lgf {

// ---------------------------------------------------------------------------
// g(x) = reunitarize(1 + Delta'(x)) in FP64 (Sec. 2 first-order expansion,
// Gram-Schmidt on rows 1-2, row 3 = (a x b)^* as in Sec. 3.2)
// ---------------------------------------------------------------------------

// f0 = (Im D11, Im D22), f1 = D12, f2 = D13, f3 = D23 of the filtered field.
// Rows of 1 + X: r1 = (1 + i a, f1, f2) and r2 = (-conj f1, 1 + i d, f3)
// with a = Re f0, d = Im f0.  Gram-Schmidt: u = r1 / |r1| and
// v = w / |w| with w = r2 - <u, r2> u = r2 - (c / |r1|^2) r1, where
// c = <r1, r2> = sum_j conj(r1_j) r2_j = (a + d)(Im f1 + i Re f1) + conj(f2) f3
// (the two terms in f1 combine).  All of it in FP64.
// The FP64 Gram-Schmidt factors of 1 + X: i1 = 1/|r1|, w = r2 - k r1 and
// i2 = 1/|w|, so that u = i1 r1 and v = i2 w.
struct GSFactors {
  double i1, i2;
  double2 w[3];
};

__device__ __forceinline__ void gram_schmidt_factors(double a, double d, double2 f1, double2 f2, double2 f3,
                                                     GSFactors& o) {
  const double n1 = fma(f2.x, f2.x, fma(f2.y, f2.y, fma(f1.x, f1.x, fma(f1.y, f1.y, fma(a, a, 1.0)))));
  o.i1 = rsqrt_fp64(n1);
  const double s = a + d;
  const double q = o.i1 * o.i1;  // 1 / |r1|^2
  const double kx = q * fma(f2.x, f3.x, fma(f2.y, f3.y, s * f1.y));
  const double ky = q * fma(f2.x, f3.y, fma(-f2.y, f3.x, s * f1.x));
  // w = r2 - k r1
  o.w[0] = make_double2(fma(ky, a, -f1.x - kx), fma(-kx, a, f1.y - ky));
  o.w[1] = make_double2(fma(ky, f1.y, fma(-kx, f1.x, 1.0)), fma(-ky, f1.x, fma(-kx, f1.y, d)));
  o.w[2] = make_double2(fma(ky, f2.y, fma(-kx, f2.x, f3.x)), fma(-ky, f2.x, fma(-kx, f2.y, f3.y)));
  const double n2 = fma(o.w[2].x, o.w[2].x, fma(o.w[2].y, o.w[2].y, fma(o.w[1].x, o.w[1].x,
                    fma(o.w[1].y, o.w[1].y, fma(o.w[0].x, o.w[0].x, o.w[0].y * o.w[0].y)))));
  o.i2 = rsqrt_fp64(n2);
}

// The FP64 factors for fields stored in FP32: i1 = 1/|r1|, the projection
// coefficient k = <r1, r2>/|r1|^2 and i2 = 1/|w| with w = r2 - k r1, where
// |w|^2 = |r2|^2 - |<r1, r2>|^2/|r1|^2 (Pythagoras for the projection) is
// formed from the inputs, so that w itself is never needed in FP64: the
// FP32 field applies k in FP32.  The singular values of 1 + X, X anti-Hermitian,
// are at least 1, so |w| >= 1 while |r2|^2 <= 1 + 5 max|X|^2: the difference
// loses no bits for |X| < 1 and up to log2 of that ratio where large rows are
// nearly dependent.  33 FP64 operations and two estimates, against 43 when w
// is formed in FP64.  Taken by entries outside the range of the FP32 pairs below.
struct GSFactors32 {
  double i1, i2, kx, ky;
};

__device__ __forceinline__ void gram_schmidt_factors_f32(double a, double d, double2 f1, double2 f2, double2 f3,
                                                         GSFactors32& o) {
  const double n1 = fma(f2.x, f2.x, fma(f2.y, f2.y, fma(f1.x, f1.x, fma(f1.y, f1.y, fma(a, a, 1.0)))));
  o.i1 = rsqrt_fp64(n1);
  const double s = a + d;
  const double q = o.i1 * o.i1;  // 1 / |r1|^2
  const double cx = fma(f2.x, f3.x, fma(f2.y, f3.y, s * f1.y));
  const double cy = fma(f2.x, f3.y, fma(-f2.y, f3.x, s * f1.x));
  const double nr2 = fma(f3.x, f3.x, fma(f3.y, f3.y, fma(d, d, fma(f1.x, f1.x, fma(f1.y, f1.y, 1.0)))));
  const double n2 = fma(-q, fma(cx, cx, cy * cy), nr2);
  o.kx = q * cx;
  o.ky = q * cy;
  o.i2 = rsqrt_fp64(n2);
}

// FP32 <-> FP64 conversions on the integer pipe, written from the IEEE 754
// binary32 / binary64 layouts: sign, rebiased exponent and mantissa apart.
// Zero and subnormal inputs give zero; FP64 -> FP32 rounds to nearest with
// ties away from zero (IEEE rounds ties to even: the two differ only on exact
// ties) and overflows to infinity.  Non-finite values are not expected here.
__device__ __forceinline__ double f32_to_f64_int(float x) {
  const uint32_t b = __float_as_uint(x);
  const uint64_t sign = (uint64_t)(b >> 31) << 63;
  const uint32_t e = (b >> 23) & 0xffu;
  const uint64_t body = ((uint64_t)(e + (1023u - 127u)) << 52) | ((uint64_t)(b & 0x7fffffu) << 29);
  return __longlong_as_double((long long)(sign | (e == 0u ? 0ull : body)));
}
__device__ __forceinline__ float f64_to_f32_int(double x) {
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  const uint32_t sign = (uint32_t)(b >> 63) << 31;
  const int64_t r = (int64_t)(b & 0x7fffffffffffffffull) - ((int64_t)(1023 - 127) << 52) + (1ll << 28);
  uint32_t f = r <= (1ll << 28) ? 0u : (uint32_t)(r >> 29);
  if (r > (1ll << 28) && f >= 0x7f800000u) f = 0x7f800000u;
  return __uint_as_float(sign | f);
}
__device__ __forceinline__ double2 c_f32_to_f64_int(float2 v) { return make_double2(f32_to_f64_int(v.x), f32_to_f64_int(v.y)); }
__device__ __forceinline__ float2 c_f64_to_f32_int(double2 v) { return make_float2(f64_to_f32_int(v.x), f64_to_f32_int(v.y)); }

// The same factors in FP32 pairs h + l (|l| <= ulp(h)/2: 48 bits) on the FP32
// pipe, which has 64 times the FP64 rate: error-free products (FMA) and sums
// (Knuth, The Art of Computer Programming 2, 4.2.2), about 200 FP32 operations.
// Each factor is within 2^-35 of its exact value before it is rounded to FP32:
// for |X| <= GS_PAIR_MAX, over rows made to be nearly dependent, i1 within
// 2^-44.7 and i2, whose difference cancels there, 2^-43.7 at |X| <= 1, 2^-37.7
// at 8, 2^-35.6 at 16, 2^-33.2 at 32, 2^-20 at 4096.
struct Pair32 {
  float h, l;
};
__device__ __forceinline__ Pair32 two_prod(float a, float b) {
  const float h = __fmul_rn(a, b);
  return Pair32{h, __fmaf_rn(a, b, -h)};
}
__device__ __forceinline__ Pair32 two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  return Pair32{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
__device__ __forceinline__ Pair32 pair_add(Pair32 a, Pair32 b) {
  const Pair32 s = two_sum(a.h, b.h);
  return Pair32{s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l))};
}
__device__ __forceinline__ Pair32 pair_norm(Pair32 a) {  // |a.h| >= |a.l|
  const float h = __fadd_rn(a.h, a.l);
  return Pair32{h, __fsub_rn(a.l, __fsub_rn(h, a.h))};
}
// 1 / sqrt(n), n >= 1: a Newton step on the estimate, with its residual exact to 2^-44.
__device__ __forceinline__ Pair32 pair_rsqrt(Pair32 n) {
  const float y = rsqrtf(n.h);
  const Pair32 p = two_prod(y, y);
  const float r = fmaf(-n.l, p.h, fmaf(-n.h, p.l, fmaf(-n.h, p.h, 1.f)));
  const float yr = y * r;
  return Pair32{y, fmaf(0.375f * r, yr, 0.5f * yr)};
}

struct GSFactorsOut {
  float i1, i2, kx, ky;
};
// Entries beyond this, and NaN, take FP64.
constexpr float GS_PAIR_MAX = 16.f;
static __device__ __noinline__ GSFactorsOut gram_schmidt_fp64_call(float2 f0, float2 f1, float2 f2, float2 f3) {
  GSFactors32 o;
  gram_schmidt_factors_f32(f32_to_f64_int(f0.x), f32_to_f64_int(f0.y), c_f32_to_f64_int(f1), c_f32_to_f64_int(f2),
                           c_f32_to_f64_int(f3), o);
  return GSFactorsOut{f64_to_f32_int(o.i1), f64_to_f32_int(o.i2), f64_to_f32_int(o.kx), f64_to_f32_int(o.ky)};
}
__device__ __forceinline__ GSFactorsOut gram_schmidt_pair(float2 f0, float2 f1, float2 f2, float2 f3) {
  auto mag = [](float x) { return __float_as_uint(x) & 0x7fffffffu; };
  const uint32_t m = max(max(max(mag(f0.x), mag(f0.y)), max(mag(f1.x), mag(f1.y))),
                         max(max(mag(f2.x), mag(f2.y)), max(mag(f3.x), mag(f3.y))));
  if (m > __float_as_uint(GS_PAIR_MAX)) return gram_schmidt_fp64_call(f0, f1, f2, f3);
  const float a = f0.x, d = f0.y;
  const Pair32 n11 = pair_add(two_prod(f1.x, f1.x), two_prod(f1.y, f1.y));
  const Pair32 n22 = pair_add(two_prod(f2.x, f2.x), two_prod(f2.y, f2.y));
  const Pair32 n33 = pair_add(two_prod(f3.x, f3.x), two_prod(f3.y, f3.y));
  // |r1|^2 and |r2|^2
  const Pair32 n1 = pair_norm(pair_add(Pair32{1.f, 0.f}, pair_add(two_prod(a, a), pair_add(n11, n22))));
  const Pair32 nr2 = pair_add(Pair32{1.f, 0.f}, pair_add(two_prod(d, d), pair_add(n11, n33)));
  const Pair32 i1 = pair_rsqrt(n1);
  Pair32 q = two_prod(i1.h, i1.h);  // 1 / |r1|^2
  q.l = fmaf(2.f * i1.h, i1.l, q.l);
  const Pair32 s = two_sum(a, d);
  auto times_s = [&](float x) {
    Pair32 p = two_prod(s.h, x);
    p.l = fmaf(s.l, x, p.l);
    return p;
  };
  const Pair32 cx = pair_norm(pair_add(times_s(f1.y), pair_add(two_prod(f2.y, f3.y), two_prod(f2.x, f3.x))));
  const Pair32 cy = pair_norm(pair_add(times_s(f1.x), pair_add(two_prod(-f2.y, f3.x), two_prod(f2.x, f3.y))));
  auto square = [](Pair32 x) {
    Pair32 p = two_prod(x.h, x.h);
    p.l = fmaf(2.f * x.h, x.l, p.l);
    return p;
  };
  const Pair32 c2 = pair_norm(pair_add(square(cx), square(cy)));
  Pair32 t = two_prod(-q.h, c2.h);
  t.l = fmaf(-q.h, c2.l, fmaf(-q.l, c2.h, t.l));
  const Pair32 i2 = pair_rsqrt(pair_norm(pair_add(nr2, t)));
  GSFactorsOut o;
  o.i1 = i1.h + i1.l;
  o.i2 = i2.h + i2.l;
  o.kx = fmaf(q.h, cx.h, fmaf(q.h, cx.l, q.l * cx.h));
  o.ky = fmaf(q.h, cy.h, fmaf(q.h, cy.l, q.l * cy.h));
  return o;
}

// Rows u, v of g = reunitarize(1 + X) in the field precision R.  FP64 fields
// take u = i1 r1 and v = i2 w in FP64.  FP32 fields, whose rows are stored in
// FP32, round their factors to FP32: u = fl(i1) r1 with r1 the FP32 entries of
// the filtered field itself, v = fl(i2) fl(w) -- within one FP32 rounding of
// the product of the exact factors.  Pass C with those factors in FP64 sat on
// the FP64 pipe (82 % busy): in pairs 84 -> 48 us at 32^4, 754 -> 461 us at
// 48^3x96 (12-real FP32 links).
template <typename R>
__device__ __forceinline__ void gauge_rows(C2<R> f0, C2<R> f1, C2<R> f2, C2<R> f3, C2<R> u[3], C2<R> v[3]) {
  if constexpr (sizeof(R) == sizeof(double)) {
    GSFactors o;
    gram_schmidt_factors(f0.x, f0.y, f1, f2, f3, o);
    u[0] = mkc<R>(o.i1, f0.x * o.i1);
    u[1] = cscale<R>(f1, o.i1);
    u[2] = cscale<R>(f2, o.i1);
#pragma unroll
    for (int j = 0; j < 3; ++j) v[j] = cscale<double>(o.w[j], o.i2);
  } else {
    const GSFactorsOut o32 = gram_schmidt_pair(f0, f1, f2, f3);
    const float i1 = o32.i1, i2 = o32.i2, kx = o32.kx, ky = o32.ky;
    const float a = f0.x, d = f0.y;
    u[0] = mkc<R>(i1, a * i1);
    u[1] = cscale<R>(f1, i1);
    u[2] = cscale<R>(f2, i1);
    // w = r2 - k r1 in FP32
    const C2<R> w0 = mkc<R>(fmaf(ky, a, -f1.x - kx), fmaf(-kx, a, f1.y - ky));
    const C2<R> w1 = mkc<R>(fmaf(ky, f1.y, fmaf(-kx, f1.x, 1.f)), fmaf(-ky, f1.x, fmaf(-kx, f1.y, d)));
    const C2<R> w2 = mkc<R>(fmaf(ky, f2.y, fmaf(-kx, f2.x, f3.x)), fmaf(-ky, f2.x, fmaf(-kx, f2.y, f3.y)));
    v[0] = cscale<R>(w0, i2);
    v[1] = cscale<R>(w1, i2);
    v[2] = cscale<R>(w2, i2);
  }
}

// Rows 1 and 2 of g = exp(X) (the exponential of Eq. (eq:gx) evaluated
// exactly instead of to first order), for X traceless anti-Hermitian packed
// as above, followed by the same Gram-Schmidt projection.
//
// With X = iQ (Q Hermitian, traceless) the Cayley-Hamilton theorem gives
// Q^3 = u Q + w 1, u = tr(Q^2)/2, w = det Q, so exp(iQ) = c0 1 + c1 Q + c2 Q^2.
// Scaling and squaring (Moler and Van Loan, "Nineteen dubious ways to compute
// the exponential of a matrix", 1978): Z = Q / 2^s with |Z|_F <= 1/4, the
// Taylor series of exp(iZ) to order 12 (remainder below 3e-18) reduced to
// c0 + c1 Z + c2 Z^2 through Z^3 = uz Z + wz 1, then s squarings carried out on
// the three coefficients with the same reduction.
__device__ __forceinline__ void gauge_exp_from_packed(double2 f0, double2 f1, double2 f2, double2 f3, double2 u[3],
                                                      double2 v[3]) {
  const double a = f0.x, d = f0.y, q33 = -(a + d);
  // Q = -iX: off-diagonal entries q12, q13, q23; Q_ji = conj(Q_ij)
  const double2 q12 = make_double2(f1.y, -f1.x), q13 = make_double2(f2.y, -f2.x), q23 = make_double2(f3.y, -f3.x);
  const double n12 = cnorm2<double>(q12), n13 = cnorm2<double>(q13), n23 = cnorm2<double>(q23);
  const double uq = 0.5 * (a * a + d * d + q33 * q33) + n12 + n13 + n23;
  const double2 t = cconjmul<double>(q13, cmul<double>(q12, q23));  // q12 q23 conj(q13)
  const double wq = a * d * q33 + 2.0 * t.x - a * n23 - d * n13 - q33 * n12;
  int s = 0;
  double n2 = 2.0 * uq, uz = uq, wz = wq;
  while (n2 > 0.0625 && s < 64) {
    n2 *= 0.25;
    uz *= 0.25;
    wz *= 0.125;
    ++s;
  }
  // Z^n / n! = al 1 + be Z + ga Z^2 (real); exp(iZ) = sum_n i^n Z^n / n!
  double al = 1.0, be = 0.0, ga = 0.0;
  double2 c0 = make_double2(1.0, 0.0), c1 = make_double2(0.0, 0.0), c2 = make_double2(0.0, 0.0);
#pragma unroll
  for (int n = 1; n <= 12; ++n) {
    const double inv = 1.0 / (double)n;
    const double al2 = ga * wz * inv, be2 = fma(ga, uz, al) * inv, ga2 = be * inv;
    al = al2;
    be = be2;
    ga = ga2;
    const double sg = ((n & 3) < 2) ? 1.0 : -1.0;
    if (n & 1) {
      c0.y = fma(sg, al, c0.y);
      c1.y = fma(sg, be, c1.y);
      c2.y = fma(sg, ga, c2.y);
    } else {
      c0.x = fma(sg, al, c0.x);
      c1.x = fma(sg, be, c1.x);
      c2.x = fma(sg, ga, c2.x);
    }
  }
  double h1 = 1.0;
  for (int k = 0; k < s; ++k) {
    const double2 p00 = cmul<double>(c0, c0), p12 = cmul<double>(c1, c2), p01 = cmul<double>(c0, c1);
    const double2 p22 = cmul<double>(c2, c2), p02 = cmul<double>(c0, c2), p11 = cmul<double>(c1, c1);
    c0 = make_double2(fma(2.0 * wz, p12.x, p00.x), fma(2.0 * wz, p12.y, p00.y));
    c1 = make_double2(fma(wz, p22.x, fma(2.0 * uz, p12.x, 2.0 * p01.x)),
                      fma(wz, p22.y, fma(2.0 * uz, p12.y, 2.0 * p01.y)));
    c2 = make_double2(fma(uz, p22.x, fma(2.0, p02.x, p11.x)), fma(uz, p22.y, fma(2.0, p02.y, p11.y)));
    h1 *= 0.5;
  }
  c1 = cscale<double>(c1, h1);       // coefficient of Q
  c2 = cscale<double>(c2, h1 * h1);  // coefficient of Q^2
  // rows 1 and 2 of Q^2
  const double s11 = a * a + n12 + n13, s22 = n12 + d * d + n23;
  const double2 s12 = cadd<double>(cscale<double>(q12, a + d), cmulc<double>(q13, q23));  // + q13 conj(q23)
  const double2 s13 = cadd<double>(cscale<double>(q13, -d), cmul<double>(q12, q23));
  const double2 s23 = cadd<double>(cconjmul<double>(q12, q13), cscale<double>(q23, -a));  // conj(q12) q13 - a q23
  const double2 s21 = make_double2(s12.x, -s12.y);
  const double2 q21 = make_double2(q12.x, -q12.y);
  double2 r1[3], r2[3];
  r1[0] = cadd<double>(cadd<double>(c0, cscale<double>(c1, a)), cscale<double>(c2, s11));
  r1[1] = cadd<double>(cmul<double>(c1, q12), cmul<double>(c2, s12));
  r1[2] = cadd<double>(cmul<double>(c1, q13), cmul<double>(c2, s13));
  r2[0] = cadd<double>(cmul<double>(c1, q21), cmul<double>(c2, s21));
  r2[1] = cadd<double>(cadd<double>(c0, cscale<double>(c1, d)), cscale<double>(c2, s22));
  r2[2] = cadd<double>(cmul<double>(c1, q23), cmul<double>(c2, s23));
  // Gram-Schmidt: u = r1/|r1|, v = (r2 - <u,r2> u)/|.|
  const double i1 = rsqrt(cnorm2<double>(r1[0]) + cnorm2<double>(r1[1]) + cnorm2<double>(r1[2]));
#pragma unroll
  for (int j = 0; j < 3; ++j) u[j] = cscale<double>(r1[j], i1);
  double2 ip = cconjmul<double>(u[0], r2[0]);
  ip = cadd<double>(ip, cconjmul<double>(u[1], r2[1]));
  ip = cadd<double>(ip, cconjmul<double>(u[2], r2[2]));
  const double2 nip = make_double2(-ip.x, -ip.y);
#pragma unroll
  for (int j = 0; j < 3; ++j) v[j] = cfma<double>(nip, u[j], r2[j]);
  const double i2 = rsqrt(cnorm2<double>(v[0]) + cnorm2<double>(v[1]) + cnorm2<double>(v[2]));
#pragma unroll
  for (int j = 0; j < 3; ++j) v[j] = cscale<double>(v[j], i2);
}

// G(s) <- g G(s) of one site, full 3x3 in precision RG.
template <typename RG>
__device__ __forceinline__ void accumulate_gauge(int64_t V, int64_t s, const C2<RG> a[3], const C2<RG> b[3],
                                                 const C2<RG> c[3], C2<RG>* __restrict__ Gf) {
  C2<RG> Go[3][3];
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int col = 0; col < 3; ++col) Go[r][col] = Gf[(r * 3 + col) * V + s];
  const C2<RG>* rows[3] = {a, b, c};
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int col = 0; col < 3; ++col) {
      C2<RG> acc = cmul<RG>(rows[r][0], Go[0][col]);
      acc = cfma<RG>(rows[r][1], Go[1][col], acc);
      acc = cfma<RG>(rows[r][2], Go[2][col], acc);
      Gf[(r * 3 + col) * V + s] = acc;
    }
}

// Stores rows u, v (precision RG) and, where needed, row 3 = (u x v)^*, and
// G <- g G where tracked.  FP64 lanes keep g as fixed-point operands, and as FP64
// numbers where the field is near the identity (near_id).
template <typename RG, int GROWS>
__device__ __forceinline__ void store_gauge_rows(int64_t V, int64_t s, const C2<RG> a[3], const C2<RG> b[3],
                                                 C2<RG>* __restrict__ gf, C2<RG>* __restrict__ Gf, bool near_id) {
  C2<RG> c[3];
  const bool need_c = (GROWS == 3) || (Gf != nullptr);
  if (need_c) su3_third_row<RG>(a, b, c);
  if constexpr (sizeof(RG) == sizeof(double)) {
    if (near_id) fxg_store_fp64(gf, V, s, a, b, c);
    else fxg_store(gf, V, s, a, b, c);
  } else {
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      gf[(0 * 3 + j) * V + s] = a[j];
      gf[(1 * 3 + j) * V + s] = b[j];
      if (GROWS == 3) gf[(2 * 3 + j) * V + s] = c[j];
    }
  }
  if (Gf != nullptr) accumulate_gauge<RG>(V, s, a, b, c, Gf);
}

// g(x) of one site from its packed filtered field and its store (and G <- g G).
template <typename R, typename RG, int GROWS, bool EXPG>
__device__ __forceinline__ void gauge_site(C2<R> f0, C2<R> f1, C2<R> f2, C2<R> f3, int64_t V, int64_t s,
                                           C2<RG>* __restrict__ gf, C2<RG>* __restrict__ Gf, bool near_id = false) {
  static_assert(sizeof(R) == sizeof(RG), "g is stored in the precision of the divergence");
  C2<RG> a[3], b[3];
  if constexpr (EXPG) {
    double2 u[3], v[3];
    gauge_exp_from_packed(ccast<double, R>(f0), ccast<double, R>(f1), ccast<double, R>(f2), ccast<double, R>(f3),
                          u, v);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      a[j] = ccast<RG, double>(u[j]);
      b[j] = ccast<RG, double>(v[j]);
    }
  } else {
    gauge_rows<RG>(f0, f1, f2, f3, a, b);
  }
  store_gauge_rows<RG, GROWS>(V, s, a, b, gf, Gf, near_id);
}

// The FP64 path of a site: outside the fixed-point range, or near the identity.
template <bool EXPG>
static __device__ __noinline__ void gauge_site_fp64(double2 f0, double2 f1, double2 f2, double2 f3, int64_t V,
                                                    int64_t s, double2* __restrict__ gf, double2* __restrict__ Gf,
                                                    bool near_id) {
  gauge_site<double, double, 3, EXPG>(f0, f1, f2, f3, V, s, gf, Gf, near_id);
}

static __device__ __noinline__ void accumulate_gauge_fp64(int64_t V, int64_t s, const int4* __restrict__ gp,
                                                          int64_t gstride, double2* __restrict__ Gf) {
  M3<double> g;
  fxg_load(gp, gstride, g);
  accumulate_gauge<double>(V, s, g.e[0], g.e[1], g.e[2], Gf);
}

// G(s) <- g G(s) in fixed point, for the entries gp[e gstride] of g (a call:
// its operands would otherwise crowd the registers of every caller, tracked
// transform or not).  A g kept as FP64 numbers takes the FP64 product.
static __device__ __noinline__ void accumulate_gauge_fx(int64_t V, int64_t s, const int4* gp, int64_t gstride,
                                                        double2* __restrict__ Gf) {
  if (fxg_is_fp64(gp[0])) {
    accumulate_gauge_fp64(V, s, gp, gstride, Gf);
    return;
  }
  uint32_t m = 0, t = 0;
  FxC G[3][3];
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double2 v = Gf[(r * 3 + c) * V + s];
      m = fx_max(m, v);
      G[r][c] = fx_from(v);
    }
  double2 o[3][3];
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    FxC g[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) g[k] = fxg_unpack(gp[(r * 3 + k) * gstride]);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      FxAcc re = fx_zero(), im = fx_zero();
#pragma unroll
      for (int k = 0; k < 3; ++k) fx_cmac(re, im, g[k], fx_neg(g[k].y), G[k][c]);
      bool bx = true, by = true;
      const int64_t x = fx_sum60(re, t), y = fx_sum60(im, t);
      o[r][c].x = fx_to_double_int<60>(x, bx);
      o[r][c].y = fx_to_double_int<60>(y, by);
      if (!bx) o[r][c].x = fx_to_double_fp<60>(x);
      if (!by) o[r][c].y = fx_to_double_fp<60>(y);
    }
  }
  if (fx_bad(m, t)) {
    accumulate_gauge_fp64(V, s, gp, gstride, Gf);
    return;
  }
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int c = 0; c < 3; ++c) Gf[(r * 3 + c) * V + s] = o[r][c];
}

// g = reunitarize(1 + X) of one site in fixed point: A holds the components of
// (f0, f1, f2, f3) in units of 2^-58, each below 1 in magnitude.
//
// Rows are halved so that everything stays within the operand range (a
// projection does not see the scale): with r1 = (1 + i a, f1, f2)/2 and
// r2 = (-conj f1, 1 + i d, f3)/2, |r1|^2 and |r2|^2 lie in [1/4, 3/2); then
// u = r1 / |r1|, w = r2 - <u, r2> u with |w| in [1/2, 5/4) (the singular
// values of 1 + X are at least 1) and v = w / |w|; row 3 is (u x v)^*.
// <r1, r2> = (a + d)(Im f1 + i Re f1) + conj(f2) f3 as in gram_schmidt_factors.
// 66 real products on the integer pipe against 77 operations on the FP64 pipe.
__device__ __forceinline__ void gauge_site_fx(const int64_t A[8], int64_t V, int64_t s, double2* __restrict__ gf,
                                              double2* __restrict__ Gf) {
  uint32_t t = 0;  // no sum can leave the range here
  const int64_t half = (int64_t)1 << 58;
  Fx f[8];  // a, d, f1, f2, f3
#pragma unroll
  for (int k = 0; k < 8; ++k) f[k] = fx_operand(2 * A[k]);
  const FxC f1{f[2], f[3]}, f2{f[4], f[5]}, f3{f[6], f[7]};
  FxAcc n = fx_zero();
  n.hi = half;  // 1/4
  fx_mac(n, f[0], f[0]);
  fx_mac(n, f1.x, f1.x);
  fx_mac(n, f1.y, f1.y);
  fx_mac(n, f2.x, f2.x);
  fx_mac(n, f2.y, f2.y);
  const int64_t yh = fx_half_rsqrt(fx_sum60(n, t));
  const Fx y = fx_operand(yh);
  // u = 2 (y/2) r1
  auto scaled = [&](Fx a, Fx b) {
    FxAcc p = fx_zero();
    fx_mac(p, a, b);
    return 2 * fx_sum60(p, t);
  };
  FxC g[3][3];
  g[0][0] = FxC{y, fx_operand(scaled(f[0], y))};
  g[0][1] = FxC{fx_operand(scaled(f1.x, y)), fx_operand(scaled(f1.y, y))};
  g[0][2] = FxC{fx_operand(scaled(f2.x, y)), fx_operand(scaled(f2.y, y))};
  // <r1, r2>, then <u, r2>
  const Fx sm = fx_operand(2 * (A[0] + A[1]));
  FxAcc cr = fx_zero(), ci = fx_zero();
  fx_mac(cr, sm, f1.y);
  fx_mac(cr, f2.x, f3.x);
  fx_mac(cr, f2.y, f3.y);
  fx_mac(ci, sm, f1.x);
  fx_mac(ci, f2.x, f3.y);
  fx_mac(ci, fx_neg(f2.y), f3.x);
  const Fx kx = fx_operand(-scaled(fx_operand(fx_sum60(cr, t)), y));
  const Fx ky = fx_operand(-scaled(fx_operand(fx_sum60(ci, t)), y));
  const FxC k{kx, ky};  // -<u, r2>
  // w = r2 - <u, r2> u
  const int64_t r2[3][2] = {{-2 * A[2], 2 * A[3]}, {2 * half, 2 * A[1]}, {2 * A[6], 2 * A[7]}};
  FxC w[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    FxAcc re = fx_zero(), im = fx_zero();
    re.hi = r2[j][0];
    im.hi = r2[j][1];
    fx_cmac(re, im, k, fx_neg(ky), g[0][j]);
    w[j] = FxC{fx_operand(fx_sum60(re, t)), fx_operand(fx_sum60(im, t))};
  }
  n = fx_zero();
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    fx_mac(n, w[j].x, w[j].x);
    fx_mac(n, w[j].y, w[j].y);
  }
  const Fx z = fx_operand(fx_half_rsqrt(fx_sum60(n, t)));
#pragma unroll
  for (int j = 0; j < 3; ++j) g[1][j] = FxC{fx_operand(scaled(w[j].x, z)), fx_operand(scaled(w[j].y, z))};
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    FxAcc re = fx_zero(), im = fx_zero();
    fx_cross_conj(re, im, g[0][(j + 1) % 3], g[0][(j + 2) % 3], g[1][(j + 1) % 3], g[1][(j + 2) % 3]);
    g[2][j] = FxC{fx_operand(fx_sum60(re, t)), fx_operand(fx_sum60(im, t))};
  }
  int4* p = reinterpret_cast<int4*>(gf);
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int j = 0; j < 3; ++j) p[(r * 3 + j) * V + s] = fxg_pack(g[r][j]);
  if (Gf != nullptr) accumulate_gauge_fx(V, s, p + s, V, Gf);
}

}  // namespace lgf
