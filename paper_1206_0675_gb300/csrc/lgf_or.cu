// Overrelaxation Landau gauge fixing: one colour of a checkerboard sweep.
//
// arXiv:1206.0675 (Sec. 3.2) names overrelaxation as the gauge-fixing method
// that needs less memory than the Fourier-accelerated one; the method is the
// published one it refers to:
//   * local maximisation of F[g] = (1/(4 Nc V)) sum Re Tr g(x) U_mu(x)
//     g^dag(x + mu^) (Sec. 2) one site at a time, all sites of one
//     checkerboard colour at once (no site has a neighbour of its own colour);
//   * Cabibbo and Marinari (Phys. Lett. B 119 (1982) 387): the SU(3)
//     maximisation in the SU(2) subgroups (0,1), (0,2), (1,2) in turn;
//   * Mandula and Ogilvie (Phys. Lett. B 248 (1990) 156): each SU(2)
//     maximiser r replaced by r^omega ~ 1 + omega (r - 1), 1 <= omega < 2,
//     projected back onto SU(2).
// At a site x of the colour, w(x) = sum_mu [U_mu(x) + U_mu^dag(x - mu^)]; the
// hit gives g(x), and then U_mu(x) <- g(x) U_mu(x), U_mu(x - mu^) <-
// U_mu(x - mu^) g^dag(x) and, when the transform is tracked, G(x) <- g(x) G(x).
// Every link joins two sites of opposite colour, so within one colour each
// link is read and written by exactly one thread: the update is in place.
//
// FP32 links: one thread per site of the colour.  12-real links: its eight links
// loaded at once (48 loads in flight) and kept in registers from w to the
// products, at 168 registers and 12 warps per SM.  Reading them one by one, and
// again for the products, left the warps waiting for loads (14 of 19 cycles
// between instructions): 32^4 188 -> 148 us a sweep (118 us for its bytes at
// 6.8 TB/s), 16^4 20.4 -> 16.4 us; at 128 registers 210 us, at 255 170 us.  18-real
// links do not fit 168 registers (284 bytes of spills), so theirs are read again,
// at 82 registers: 32^4 267 us against 275 kept, 24^4 87 against 91, 16^3x32 41
// against 45.  The site algebra runs in the link precision; rows 1-2 of every
// product are formed and row 3 is rebuilt as (a x b)^* (Sec. 3.2), as in the
// Fourier-accelerated update.
#include <cmath>

#include "lgf_fixed.cuh"
#include "lgf_gauge.cuh"
#include "lgf_internal.h"

namespace lgf {

constexpr int OR_THREADS = 128;

// 1/sqrt(x) in the lane precision for x > 0 (FP32: the hardware estimate and
// one Newton step).
template <typename R> __device__ __forceinline__ R or_rsqrt(R x);
template <> __device__ __forceinline__ double or_rsqrt<double>(double x) { return rsqrt_fp64(x); }
template <> __device__ __forceinline__ float or_rsqrt<float>(float x) {
  const float y = rsqrtf(x);
  return y * fmaf(-0.5f * x * y, y, 1.5f);
}

// Overrelaxed SU(2) element of one subgroup from its 2x2 block
// B = [[mii, mij], [mji, mjj]] of the running local field.  In quaternion
// form B contributes Re Tr(r B) = 2 (r0 b0 - r1 b1 - r2 b2 - r3 b3) with
// b0 = Re(B00 + B11)/2, b1 = Im(B01 + B10)/2, b2 = Re(B01 - B10)/2,
// b3 = Im(B00 - B11)/2, largest at r = (b0, -b1, -b2, -b3)/|b| (the common
// factor 1/2 drops out); r = 1 where |b|^2 is below the smallest normal
// number.  q = (1 - omega) + omega r, normalised (|q| >= 1 for omega >= 1).
// Result as the matrix [[a, b], [-conj(b), conj(a)]], a = q0 + i q3,
// b = q2 + i q1.
template <typename R>
__device__ __forceinline__ void or_subgroup(C2<R> mii, C2<R> mij, C2<R> mji, C2<R> mjj, R omega, C2<R>& a,
                                            C2<R>& b) {
  const R b0 = mii.x + mjj.x, b1 = mij.y + mji.y, b2 = mij.x - mji.x, b3 = mii.y - mjj.y;
  const R n2 = fma(b0, b0, fma(b1, b1, fma(b2, b2, b3 * b3)));
  const R tiny = sizeof(R) == sizeof(double) ? (R)2.2250738585072014e-308 : (R)1.17549435e-38f;
  R r0 = 1, r1 = 0, r2 = 0, r3 = 0;
  if (n2 >= tiny) {
    const R inv = or_rsqrt<R>(n2);
    r0 = b0 * inv;
    r1 = -b1 * inv;
    r2 = -b2 * inv;
    r3 = -b3 * inv;
  }
  const R q0 = fma(omega, r0, (R)1 - omega), q1 = omega * r1, q2 = omega * r2, q3 = omega * r3;
  const R iq = or_rsqrt<R>(fma(q0, q0, fma(q1, q1, fma(q2, q2, q3 * q3))));
  a = mkc<R>(q0 * iq, q3 * iq);
  b = mkc<R>(q2 * iq, q1 * iq);
}

// (xi, xj) <- [[a, b], [-conj(b), conj(a)]] (xi, xj): one column of the two
// rows a subgroup acts on.
template <typename R> __device__ __forceinline__ void or_rot(C2<R> a, C2<R> b, C2<R>& xi, C2<R>& xj) {
  const C2<R> ni = cfma<R>(b, xj, cmul<R>(a, xi));
  const C2<R> nj = csub<R>(cconjmul<R>(a, xj), cconjmul<R>(b, xi));
  xi = ni;
  xj = nj;
}

// g(x) of one Cabibbo-Marinari hit on the local field M (M is consumed).
template <typename R> __device__ __forceinline__ void or_site_gauge(M3<R>& M, R omega, M3<R>& gx) {
  C2<R> a, b;
  // subgroup (0, 1): g = R01 embedded; rows 0 and 1 of M rotated
  or_subgroup<R>(M.e[0][0], M.e[0][1], M.e[1][0], M.e[1][1], omega, a, b);
  gx.e[0][0] = a;
  gx.e[0][1] = b;
  gx.e[0][2] = mkc<R>(0, 0);
  gx.e[1][0] = mkc<R>(-b.x, b.y);
  gx.e[1][1] = cconj<R>(a);
  gx.e[1][2] = mkc<R>(0, 0);
  gx.e[2][0] = mkc<R>(0, 0);
  gx.e[2][1] = mkc<R>(0, 0);
  gx.e[2][2] = mkc<R>(1, 0);
#pragma unroll
  for (int c = 0; c < 3; ++c) or_rot<R>(a, b, M.e[0][c], M.e[1][c]);
  // subgroup (0, 2): rows 0 and 2 of g; of M only row 2's columns 1 and 2
  // are read again
  or_subgroup<R>(M.e[0][0], M.e[0][2], M.e[2][0], M.e[2][2], omega, a, b);
#pragma unroll
  for (int c = 0; c < 3; ++c) or_rot<R>(a, b, gx.e[0][c], gx.e[2][c]);
#pragma unroll
  for (int c = 1; c < 3; ++c) or_rot<R>(a, b, M.e[0][c], M.e[2][c]);
  // subgroup (1, 2): rows 1 and 2 of g
  or_subgroup<R>(M.e[1][1], M.e[1][2], M.e[2][1], M.e[2][2], omega, a, b);
#pragma unroll
  for (int c = 0; c < 3; ++c) or_rot<R>(a, b, gx.e[1][c], gx.e[2][c]);
}

// x - mu^ with periodic wrap, for a direction mu known only at run time:
// selects instead of indexed arrays, so that coordinates and geometry stay in
// registers (no local-memory frame in the loops over mu).
__device__ __forceinline__ int64_t or_back(const Geom& g, int64_t s, const int c[4], int mu) {
  int cm = c[0], L = g.L[0];
  int64_t st = 1;
  if (mu == 1) { cm = c[1]; L = g.L[1]; st = g.stride[1]; }
  if (mu == 2) { cm = c[2]; L = g.L[2]; st = g.stride[2]; }
  if (mu == 3) { cm = c[3]; L = g.L[3]; st = g.stride[3]; }
  return cm == 0 ? s + (int64_t)(L - 1) * st : s - st;
}

// Site j of the colour: x = 2 xh + ((y + z + t + parity) & 1) in its (y, z, t)
// row; dhx divides by Lx / 2.
__device__ __forceinline__ int64_t or_coords(const Geom& g, const FastDiv& dhx, uint32_t j, int parity, int c[4]) {
  const uint32_t row = dhx.div(j);
  const uint32_t r2 = g.dL[1].div(row);
  c[1] = (int)(row - r2 * g.dL[1].d);
  c[3] = (int)g.dL[2].div(r2);
  c[2] = (int)(r2 - (uint32_t)c[3] * g.dL[2].d);
  c[0] = 2 * (int)(j - row * dhx.d) + ((c[1] + c[2] + c[3] + parity) & 1);
  return (int64_t)c[0] + (int64_t)g.L[0] * row;
}

// The stored rows of a matrix.
template <typename R, int ROWS> struct Rows {
  C2<R> e[ROWS][3];
  // rows 1 to 3, the third rebuilt where it is not stored
  __device__ __forceinline__ void full(C2<R> (&o)[3][3]) const {
#pragma unroll
    for (int i = 0; i < ROWS; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) o[i][j] = e[i][j];
    if (ROWS == 2) su3_third_row<R>(o[0], o[1], o[2]);
  }
};
template <typename R, int ROWS>
__device__ __forceinline__ Rows<R, ROWS> load_rows(const MatField<R, ROWS>& F, int m, int64_t s) {
  Rows<R, ROWS> v;
#pragma unroll
  for (int r = 0; r < ROWS; ++r)
#pragma unroll
    for (int j = 0; j < 3; ++j) v.e[r][j] = F.p[F.off(m, r, j, s)];
  return v;
}

// w(x) = sum_mu [U_mu(x) + U_mu^dag(x - mu^)]
template <typename R, int ROWS>
__device__ __forceinline__ void or_local_field(const Geom& g, const MatField<R, ROWS>& U, const int c[4], int64_t s,
                                               M3<R>& M) {
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int k = 0; k < 3; ++k) M.e[r][k] = mkc<R>(0, 0);
#pragma unroll 1
  for (int mu = 0; mu < 4; ++mu) {
    M3<R> u;
    U.load(mu, s, u);
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int k = 0; k < 3; ++k) M.e[r][k] = cadd<R>(M.e[r][k], u.e[r][k]);
    U.load(mu, or_back(g, s, c, mu), u);
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int k = 0; k < 3; ++k) M.e[r][k] = cadd<R>(M.e[r][k], cconj<R>(u.e[k][r]));
  }
}

// U_mu(x) <- g U_mu(x): rows 0, 1 by products, row 2 = (row0 x row1)^*
template <typename R, int ROWS>
__device__ __forceinline__ void or_own_link(const MatField<R, ROWS>& U, int mu, int64_t s, const M3<R>& gx,
                                            const C2<R> (&f)[3][3]) {
  M3<R> o;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      C2<R> acc = cmul_fx<R>(gx.e[i][0], f[0][k]);
      acc = cfma<R>(gx.e[i][1], f[1][k], acc);
      o.e[i][k] = cfma<R>(gx.e[i][2], f[2][k], acc);
    }
  su3_third_row<R>(o.e[0], o.e[1], o.e[2]);
  U.store(mu, s, o);
}
// U_mu(x - mu^) <- U_mu(x - mu^) g^dag: rows 0, 1 of the old link suffice
template <typename R, int ROWS>
__device__ __forceinline__ void or_back_link(const MatField<R, ROWS>& U, int mu, int64_t sb, const M3<R>& gx,
                                             const C2<R> (*b)[3]) {
  M3<R> o;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      C2<R> acc = cmulc_fx<R>(b[i][0], gx.e[k][0]);
      acc = cfmac<R>(b[i][1], gx.e[k][1], acc);
      o.e[i][k] = cfmac<R>(b[i][2], gx.e[k][2], acc);
    }
  su3_third_row<R>(o.e[0], o.e[1], o.e[2]);
  U.store(mu, sb, o);
}
// G(x) <- g(x) G(x), full 3x3
template <typename R>
__device__ __forceinline__ void or_transform(C2<R>* __restrict__ G, int64_t V, int64_t s, const M3<R>& gx) {
  if (G == nullptr) return;
  const MatField<R, 3> Gf{G, V};
  M3<R> Go, Gn;
  Gf.load(0, s, Go);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      C2<R> acc = cmul<R>(gx.e[i][0], Go.e[0][k]);
      acc = cfma<R>(gx.e[i][1], Go.e[1][k], acc);
      Gn.e[i][k] = cfma<R>(gx.e[i][2], Go.e[2][k], acc);
    }
  Gf.store(0, s, Gn);
}

// One site of the colour: its hit and the products with its eight links, which
// stay in registers from one use to the other (of the links that end in the
// site, rows 1 and 2).
template <typename R, int ROWS>
__device__ __forceinline__ void or_site(const Geom& g, const MatField<R, ROWS>& U, const int c[4], int64_t s,
                                        C2<R>* __restrict__ G, R omega) {
  Rows<R, ROWS> u[4], b[4];
  uint32_t sb[4];  // site indices have 28 bits
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    sb[mu] = (uint32_t)or_back(g, s, c, mu);
    u[mu] = load_rows(U, mu, s);
    b[mu] = load_rows(U, mu, sb[mu]);
  }
  M3<R> M;
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int k = 0; k < 3; ++k) M.e[r][k] = mkc<R>(0, 0);
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    C2<R> f[3][3];
    u[mu].full(f);
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int k = 0; k < 3; ++k) M.e[r][k] = cadd<R>(M.e[r][k], f[r][k]);
    b[mu].full(f);
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int k = 0; k < 3; ++k) M.e[r][k] = cadd<R>(M.e[r][k], cconj<R>(f[k][r]));
  }
  M3<R> gx;
  or_site_gauge<R>(M, omega, gx);
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    C2<R> f[3][3];
    u[mu].full(f);
    or_own_link<R, ROWS>(U, mu, s, gx, f);
    or_back_link<R, ROWS>(U, mu, sb[mu], gx, b[mu].e);
  }
  or_transform<R>(G, g.V, s, gx);
}

// The same with the links read again for the products (18-real links).
template <typename R, int ROWS>
__device__ __forceinline__ void or_site_reread(const Geom& g, const MatField<R, ROWS>& U, const int c[4], int64_t s,
                                               C2<R>* __restrict__ G, R omega) {
  M3<R> M, gx;
  or_local_field<R, ROWS>(g, U, c, s, M);
  or_site_gauge<R>(M, omega, gx);
#pragma unroll 1
  for (int mu = 0; mu < 4; ++mu) {
    M3<R> u;
    U.load(mu, s, u);
    or_own_link<R, ROWS>(U, mu, s, gx, u.e);
    const int64_t sb = or_back(g, s, c, mu);
    C2<R> b[2][3];
    U.load_rows01(mu, sb, b);
    or_back_link<R, ROWS>(U, mu, sb, gx, b);
  }
  or_transform<R>(G, g.V, s, gx);
}

template <typename R, int ROWS>
__global__ void __launch_bounds__(OR_THREADS, ROWS == 3 ? 4 : 3)
or_half_sweep_kernel(Geom g, C2<R>* __restrict__ U0, C2<R>* __restrict__ U1, const DevState* __restrict__ st,
                     C2<R>* __restrict__ G, int parity, FastDiv dhx, R omega) {
  // fused FP32 lanes keep their current links in one of two buffers
  const MatField<R, ROWS> U{(U1 != nullptr && st->ubuf) ? U1 : U0, g.V};
  const uint32_t j = blockIdx.x * blockDim.x + threadIdx.x;
  if ((int64_t)j >= (g.V >> 1)) return;
  int c[4];
  const int64_t s = or_coords(g, dhx, j, parity, c);
  if (ROWS == 3) or_site_reread<R, ROWS>(g, U, c, s, G, omega);
  else or_site<R, ROWS>(g, U, c, s, G, omega);
}

// ---------------------------------------------------------------------------
// FP64 links in fixed point (lgf_fixed.cuh)
// ---------------------------------------------------------------------------
//
// Two kernels per colour: the first forms w(x) and g(x) of the colour's sites,
// one thread each; the second multiplies every link of the lattice by the one
// g that touches it, one thread per link, as in update_fx_kernel.  Warps with
// links near the identity, sites and links outside the fixed-point range, and
// local fields too small for their direction to be resolved are done in FP64.
// With FP64 arithmetic, one thread a site for all of it, the FP64 pipe was 93 %
// busy (1199 operations a site and sweep).  One fixed-point kernel with the
// hits between two barriers left three of four warps waiting for them.
// A sweep, us (FP64 arithmetic before): 18-real 24^4 329 (724), 32^4 939 (2142),
// 16^4 79 (168), 8^4 38 (93); 12-real 32^4 804 (2311).  theta of 8^4 levels off
// (omega = 1.7) at 1.1e-32 (FP64: 1.2e-31) for eps = 0.5, 3.4e-33 (2.8e-32) for 0.25,
// 3e-33 (6e-33) for 0.12; with operands of w / 64 and of r in [1/4, 1/2) it was
// 2e-31 for all of them, and a sweep 2 % shorter.  The CTAs per SM are the
// best of 3 to 6 for each kernel and storage (links of 18 reals at 4: 960 us, at 3:
// 1056).

// The 64-bit sum an operand stands for (units of 2^-60).
__device__ __forceinline__ int64_t fx_r60(Fx a) { return mad_wide(a.h, 1 << 30, (int64_t)a.l); }

// Leading zeros of the largest magnitude of four integers.
__device__ __forceinline__ int fx_lz4(const int64_t v[4]) {
  uint64_t mag = 1u;
#pragma unroll
  for (int k = 0; k < 4; ++k) mag |= (uint64_t)(v[k] < 0 ? -v[k] : v[k]);
  return __clzll((long long)mag);
}

// v / |v| of four integers, lz = fx_lz4(v).  The components are shifted to where
// an operand is finest, the largest to [1/2, 1) (UP: from below 9/8, which stays
// as it is; otherwise from [2^59, 2^63) down): |v|^2 is then in [1/4, 5.1) and
// 1 / (2 |v|) in (1/5, 1].  Every rounding here turns g(x), and theta of a
// converged field is the square of that.
template <bool UP> __device__ __forceinline__ void fx_unit4(const int64_t v[4], int lz, Fx u[4]) {
  uint32_t t = 0;
  Fx r[4];
  FxAcc n = fx_zero();
  const int sh = UP ? max(lz - 4, 0) : 4 - lz;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    r[k] = fx_operand(UP ? v[k] << sh : (v[k] + ((1 << sh) >> 1)) >> sh);
    fx_mac(n, r[k], r[k]);
  }
  const Fx y = fx_operand(fx_half_rsqrt(max(fx_sum60(n, t) >> 2, (int64_t)1 << 56)) >> 1);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    FxAcc p = fx_zero_x2();
    fx_mac(p, r[k], y);
    u[k] = fx_operand(fx_sum60_x2(p));
  }
}

// or_subgroup in fixed point, on blocks of the local field over 16 (components
// up to 9/16, their sums up to 9/8).  q is scaled by 7/16, which puts |q| in
// [0.43, 1.32) for 1 <= omega < 2: w7 = 7 omega / 16 and c7 = 7 (1 - omega) / 16
// in units of 2^-60.  ok = false where no component of b / 16 reaches 2^-21
// (|b| < 2^-17): too small for its direction to be resolved in units of 2^-60.
__device__ __forceinline__ void or_subgroup_fx(const FxC& mii, const FxC& mij, const FxC& mji, const FxC& mjj, Fx w7,
                                               int64_t c7, FxC& a, FxC& b, bool& ok) {
  const int64_t v[4] = {fx_r60(mii.x) + fx_r60(mjj.x), -(fx_r60(mij.y) + fx_r60(mji.y)),
                        fx_r60(mji.x) - fx_r60(mij.x), fx_r60(mjj.y) - fx_r60(mii.y)};  // |b| r / |r|
  const int lz = fx_lz4(v);
  ok = ok && lz <= 24;
  Fx r[4];
  fx_unit4<true>(v, lz, r);
  int64_t q[4];  // units of 2^-62: the largest component is at least 7/32, above 2^59
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    FxAcc p = fx_zero_x4();
    if (k == 0) p.hi = c7;
    fx_mac(p, w7, r[k]);
    q[k] = fx_sum60_x4(p);
  }
  fx_unit4<false>(q, fx_lz4(q), r);
  a = FxC{r[0], r[3]};
  b = FxC{r[2], r[1]};
}

// or_rot in fixed point.
__device__ __forceinline__ void or_rot_fx(const FxC& a, const FxC& b, FxC& xi, FxC& xj) {
  uint32_t t = 0;
  FxAcc ir = fx_zero(), ii = fx_zero(), jr = fx_zero(), ji = fx_zero();
  fx_cmac(ir, ii, a, fx_neg(a.y), xi);
  fx_cmac(ir, ii, b, fx_neg(b.y), xj);
  const FxC ac = fx_conj(a), nbc{fx_neg(b.x), b.y};  // conj(a), -conj(b)
  fx_cmac(jr, ji, ac, a.y, xj);
  fx_cmac(jr, ji, nbc, fx_neg(b.y), xi);
  xi = FxC{fx_operand(fx_sum60(ir, t)), fx_operand(fx_sum60(ii, t))};
  xj = FxC{fx_operand(fx_sum60(jr, t)), fx_operand(fx_sum60(ji, t))};
}

// g(x) of one Cabibbo-Marinari hit, as or_site_gauge.
__device__ __forceinline__ void or_site_gauge_fx(FxC M[3][3], Fx w7, int64_t c7, FxC gx[3][3], bool& ok) {
  const FxC zero{{0, 0}, {0, 0}}, one{{1 << 30, 0}, {0, 0}};
  FxC a, b;
  or_subgroup_fx(M[0][0], M[0][1], M[1][0], M[1][1], w7, c7, a, b, ok);
  gx[0][0] = a;
  gx[0][1] = b;
  gx[0][2] = zero;
  gx[1][0] = FxC{fx_neg(b.x), b.y};
  gx[1][1] = fx_conj(a);
  gx[1][2] = zero;
  gx[2][0] = zero;
  gx[2][1] = zero;
  gx[2][2] = one;
#pragma unroll
  for (int c = 0; c < 3; ++c) or_rot_fx(a, b, M[0][c], M[1][c]);
  or_subgroup_fx(M[0][0], M[0][2], M[2][0], M[2][2], w7, c7, a, b, ok);
#pragma unroll
  for (int c = 0; c < 3; ++c) or_rot_fx(a, b, gx[0][c], gx[2][c]);
#pragma unroll
  for (int c = 1; c < 3; ++c) or_rot_fx(a, b, M[0][c], M[2][c]);
  or_subgroup_fx(M[1][1], M[1][2], M[2][1], M[2][2], w7, c7, a, b, ok);
#pragma unroll
  for (int c = 0; c < 3; ++c) or_rot_fx(a, b, gx[1][c], gx[2][c]);
}

// g(x) of a site from FP64 sums, and its store.
template <int ROWS>
static __device__ __noinline__ void or_gauge_fp64(const Geom& g, MatField<double, ROWS> U, int64_t s,
                                                  double2* __restrict__ gf, double omega) {
  int c[4];
  site_coords(g, s, c);
  M3<double> M, gx;
  or_local_field<double, ROWS>(g, U, c, s, M);
  or_site_gauge<double>(M, omega, gx);
  fxg_store_fp64(gf, g.V, s, gx.e[0], gx.e[1], gx.e[2]);
}

template <int ROWS>
__global__ void __launch_bounds__(OR_THREADS, ROWS == 3 ? 5 : 4)
or_gauge_fx_kernel(Geom g, MatField<double, ROWS> U, double2* __restrict__ gf, double2* __restrict__ G, int parity,
                   FastDiv dhx, double omega, int64_t w7, int64_t c7) {
  const uint32_t j0 = blockIdx.x * blockDim.x + threadIdx.x, n = (uint32_t)(g.V >> 1);
  const bool in = j0 < n;
  int c[4];
  const int64_t s = or_coords(g, dhx, in ? j0 : n - 1, parity, c);  // lanes past the end follow their warp
  // w(x) in units of 2^-59
  int64_t W[9][2];
#pragma unroll
  for (int e = 0; e < 9; ++e) W[e][0] = W[e][1] = 0;
  uint32_t m = 0, t = 0;
  // before the loop: a way out of it costs the loads' order (32^4 957 -> 939 us a sweep)
  const bool near_id = __any_sync(
      0xffffffffu, fx_max(fx_max(fx_max(0u, __ldg(&U.p[U.off(0, 0, 1, s)])), __ldg(&U.p[U.off(0, 0, 2, s)])),
                          __ldg(&U.p[U.off(0, 1, 2, s)])) < FX_NEAR_HI);
  if (near_id) {
    if (!in) return;
    or_gauge_fp64<ROWS>(g, U, s, gf, omega);
    if (G != nullptr) accumulate_gauge_fp64(g.V, s, reinterpret_cast<const int4*>(gf) + s, g.V, G);
    return;
  }
#pragma unroll 1
  for (int k = 0; k < 8; ++k) {
    const int mu = k >> 1;
    const bool fwd = (k & 1) == 0;
    const int64_t sl = fwd ? s : or_back(g, s, c, mu);
    double2 u[ROWS][3];
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
#pragma unroll
      for (int q = 0; q < 3; ++q) u[r][q] = __ldg(&U.p[U.off(mu, r, q, sl)]);
    int64_t x[3][3][2];
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        m = fx_max(m, u[r][q]);
        x[r][q][0] = fxk_from<59>(u[r][q].x);
        x[r][q][1] = fxk_from<59>(u[r][q].y);
      }
    if (ROWS == 2) {
      FxC a[2][3];
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int q = 0; q < 3; ++q) a[r][q] = FxC{fx_operand(2 * x[r][q][0]), fx_operand(2 * x[r][q][1])};
      int64_t c3[3][2];
      fx_third_row(a[0], a[1], c3, t);
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        x[2][q][0] = c3[q][0] >> 1;
        x[2][q][1] = c3[q][1] >> 1;
      }
    }
    if (fwd) {
#pragma unroll
      for (int e = 0; e < 9; ++e) {
        W[e][0] += x[e / 3][e % 3][0];
        W[e][1] += x[e / 3][e % 3][1];
      }
    } else {
#pragma unroll
      for (int e = 0; e < 9; ++e) {
        W[e][0] += x[e % 3][e / 3][0];
        W[e][1] -= x[e % 3][e / 3][1];
      }
    }
  }
  FxC M[3][3], gx[3][3];
#pragma unroll
  for (int e = 0; e < 9; ++e) M[e / 3][e % 3] = FxC{fx_operand((W[e][0] + 4) >> 3), fx_operand((W[e][1] + 4) >> 3)};  // w / 16
  bool ok = !fx_bad(m, t);
  or_site_gauge_fx(M, fx_operand(w7), c7, gx, ok);
  if (!in) return;
  if (ok) {
    int4* p = reinterpret_cast<int4*>(gf);
#pragma unroll
    for (int e = 0; e < 9; ++e) p[e * g.V + s] = fxg_pack(gx[e / 3][e % 3]);
  } else {
    or_gauge_fp64<ROWS>(g, U, s, gf, omega);
  }
  if (G != nullptr) accumulate_gauge_fx(g.V, s, reinterpret_cast<const int4*>(gf) + s, g.V, G);
}

// One link in FP64: fwd ? g U : U g^dag (of which rows 1-2 of the old link suffice).
template <int ROWS>
static __device__ __noinline__ void or_link_fp64(MatField<double, ROWS> U, const double2* gf, int mu, int64_t sl,
                                                 int64_t s, bool fwd) {
  M3<double> g, u, o;
  fxg_load(gf, U.V, s, g);
  if (fwd) {
    U.load(mu, sl, u);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        double2 acc = cmul_fx<double>(g.e[i][0], u.e[0][k]);
        acc = cfma<double>(g.e[i][1], u.e[1][k], acc);
        o.e[i][k] = cfma<double>(g.e[i][2], u.e[2][k], acc);
      }
  } else {
    U.load_rows01(mu, sl, u.e);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        double2 acc = cmulc_fx<double>(u.e[i][0], g.e[k][0]);
        acc = cfmac<double>(u.e[i][1], g.e[k][1], acc);
        o.e[i][k] = cfmac<double>(u.e[i][2], g.e[k][2], acc);
      }
  }
  su3_third_row<double>(o.e[0], o.e[1], o.e[2]);
  U.store(mu, sl, o);
}

// A CTA takes 32 sites of the colour and half of their links: four warps, the
// directions' forward (even blockIdx.x) or backward links.  The sites of a colour
// use half of every 32-byte sector; the other half belongs to backward links of
// neighbouring rows, so the two kinds alternate and the sector is still in L2
// (all forward links first: 77 % of the DRAM bandwidth, 394 against 324 us a
// sweep of 24^4).
template <int ROWS>
__global__ void __launch_bounds__(OR_THREADS, 5)
or_links_fx_kernel(Geom g, MatField<double, ROWS> U, const double2* __restrict__ gf, int parity, FastDiv dhx) {
  const uint32_t j0 = (blockIdx.x >> 1) * 32u + (threadIdx.x & 31u), nc = (uint32_t)(g.V >> 1);
  const bool in = j0 < nc;
  const int mu = threadIdx.x >> 5;
  const bool fwd = (blockIdx.x & 1u) == 0;
  int c[4];
  const int64_t s = or_coords(g, dhx, in ? j0 : nc - 1, parity, c);  // lanes past the end follow their warp
  const int64_t sl = fwd ? s : or_back(g, s, c, mu);
  const int4* p = reinterpret_cast<const int4*>(gf);
  constexpr int UR = ROWS;
  double2 u[UR][3];
  int4 g4[3][3];
#pragma unroll
  for (int r = 0; r < UR; ++r)
#pragma unroll
    for (int k = 0; k < 3; ++k) u[r][k] = U.p[U.off(mu, r, k, sl)];
#pragma unroll
  for (int e = 0; e < 9; ++e) g4[e / 3][e % 3] = __ldg(&p[e * g.V + s]);
  // as the hits' own test, so that most g in FP64 meet links that take FP64
  if (__any_sync(0xffffffffu, fx_max(fx_max(fx_max(0u, u[0][1]), u[0][2]), u[1][2]) < FX_NEAR_HI)) {
    if (in) or_link_fp64<ROWS>(U, gf, mu, sl, s, fwd);
    return;
  }
  uint32_t m = 0, t = 0;
  FxC x[3][3];
#pragma unroll
  for (int r = 0; r < UR; ++r)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      m = fx_max(m, u[r][k]);
      x[r][k] = fx_from(u[r][k]);
    }
  int64_t n[2][3][2];
  if (fwd) {
    if (ROWS == 2) {
      int64_t c3[3][2];
      fx_third_row(x[0], x[1], c3, t);
#pragma unroll
      for (int k = 0; k < 3; ++k) x[2][k] = FxC{fx_operand(c3[k][0]), fx_operand(c3[k][1])};
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        FxAcc re = fx_zero(), im = fx_zero();
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const FxC a = fxg_unpack(g4[i][q]);
          fx_cmac(re, im, a, fx_neg(a.y), x[q][k]);
        }
        n[i][k][0] = fx_sum60(re, t);
        n[i][k][1] = fx_sum60(im, t);
      }
  } else {
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        FxAcc re = fx_zero(), im = fx_zero();
#pragma unroll
        for (int q = 0; q < 3; ++q) fx_cmacc(re, im, x[i][q], fx_neg(x[i][q].x), fxg_unpack(g4[k][q]));
        n[i][k][0] = fx_sum60(re, t);
        n[i][k][1] = fx_sum60(im, t);
      }
  }
  int64_t n3[3][2];
  if (ROWS == 3) {
    FxC r[2][3];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int k = 0; k < 3; ++k) r[i][k] = FxC{fx_operand(n[i][k][0]), fx_operand(n[i][k][1])};
    fx_third_row(r[0], r[1], n3, t);
  }
  if (!in) return;
  if (fx_bad(m, t) || fxg_is_fp64(g4[0][0])) {
    or_link_fp64<ROWS>(U, gf, mu, sl, s, fwd);
    return;
  }
  double2 o[ROWS][3];
  fx_link_to_double<ROWS>(n, n3, o);
#pragma unroll
  for (int r = 0; r < ROWS; ++r)
#pragma unroll
    for (int k = 0; k < 3; ++k) U.p[U.off(mu, r, k, sl)] = o[r][k];
}

template <typename R, int ROWS>
cudaError_t launch_or_half_sweep(const Geom& g, C2<R>* U0, C2<R>* U1, const DevState* st, C2<R>* gfield, C2<R>* G,
                                 int parity, double omega, cudaStream_t s) {
  const int64_t n = g.V >> 1;
  const FastDiv dhx = FastDiv::make((uint32_t)g.L[0] / 2);
  if constexpr (sizeof(R) == sizeof(double)) {
    // FP64 lanes have one link buffer
    const int64_t w7 = std::llround(std::ldexp(7.0 * omega, 56)), c7 = std::llround(std::ldexp(7.0 * (1.0 - omega), 56));
    const MatField<double, ROWS> U{U0, g.V};
    or_gauge_fx_kernel<ROWS><<<(unsigned)((n + OR_THREADS - 1) / OR_THREADS), OR_THREADS, 0, s>>>(
        g, U, gfield, G, parity & 1, dhx, omega, w7, c7);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    or_links_fx_kernel<ROWS><<<2 * (unsigned)((n + 31) / 32), OR_THREADS, 0, s>>>(g, U, gfield, parity & 1, dhx);
  } else {
    const unsigned nb = (unsigned)((n + OR_THREADS - 1) / OR_THREADS);
    or_half_sweep_kernel<R, ROWS><<<nb, OR_THREADS, 0, s>>>(g, U0, U1, st, G, parity & 1, dhx, (R)omega);
  }
  return cudaGetLastError();
}

template cudaError_t launch_or_half_sweep<double, 3>(const Geom&, double2*, double2*, const DevState*, double2*, double2*, int,
                                                     double, cudaStream_t);
template cudaError_t launch_or_half_sweep<double, 2>(const Geom&, double2*, double2*, const DevState*, double2*, double2*, int,
                                                     double, cudaStream_t);
template cudaError_t launch_or_half_sweep<float, 3>(const Geom&, float2*, float2*, const DevState*, float2*, float2*, int,
                                                    double, cudaStream_t);
template cudaError_t launch_or_half_sweep<float, 2>(const Geom&, float2*, float2*, const DevState*, float2*, float2*, int,
                                                    double, cudaStream_t);

}  // namespace lgf
