// Roots of unity in fixed point for the integer transform passes (host code).
#pragma once

#include <cmath>

namespace lgf {

// The roots exp(-2 pi i m / N), m < N <= 128, as limbs: hl[4 m] to hl[4 m + 3]
// are h and l of the cosine, then of the sine, each h 2^-30 + l 2^-60 with both
// rounded to nearest.  Returns how many angles were evaluated.
//
// Every angle is one of [0, pi/4] reflected into its octant, and the limbs of a
// reflected root are those of the angle, exchanged or negated: N / 8 + 1
// evaluations for a multiple of 8, N / 2 + 1 for an odd N.  long double is
// 128-bit software arithmetic on aarch64, where 2 N evaluations per direction
// took up to 150 us of lgf_create (81x2x2x128).
inline int fixed_roots(int N, int* hl) {
  const long double two_pi = 6.283185307179586476925286766559005768L;
  struct Angle {
    int h[2], l[2];  // cosine and sine
    bool known;
  } angle[129] = {};
  int evaluated = 0;
  for (int m = 0; m < N; ++m) {
    const int o = 8 * m / N, r = 8 * m - o * N;
    const int j = (o & 1) ? N - r : r;  // the angle is 2 pi j / (8 N)
    Angle& a = angle[j];
    if (!a.known) {
      const long double t = two_pi * (long double)j / (long double)(8 * N);
      const long double c[2] = {std::cos(t), std::sin(t)};
      for (int k = 0; k < 2; ++k) {
        const long double h = std::round(c[k] * 1073741824.0L);
        a.h[k] = (int)h;
        a.l[k] = (int)std::round((c[k] * 1073741824.0L - h) * 1073741824.0L);
      }
      a.known = true;
      ++evaluated;
    }
    // cosine and sine exchange in octants 1, 2, 5 and 6; the cosine is negative
    // in octants 2 to 5, the sine (of the positive angle) in octants 4 to 7
    const int swap = ((o + 1) >> 1) & 1, nc = (o >= 2 && o <= 5) ? -1 : 1, ns = o >= 4 ? 1 : -1;
    hl[4 * m] = nc * a.h[swap];
    hl[4 * m + 1] = nc * a.l[swap];
    hl[4 * m + 2] = ns * a.h[swap ^ 1];
    hl[4 * m + 3] = ns * a.l[swap ^ 1];
  }
  return evaluated;
}

}  // namespace lgf
