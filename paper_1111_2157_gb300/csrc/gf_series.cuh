// Chebyshev series of a resolvent 1 / (z - e) in e (device code only): band sums of many frequencies
// from one set of moments, for the block form and the pole path's G_loc.
#pragma once

#include "gf_complex.cuh"
#include "gf_gj64.cuh"

namespace gf {
namespace series {

using namespace cx;

// Coefficients of the Chebyshev series at z (x = (z - c) / r, s = sqrt(x^2 - 1), xi = x - s):
//   1/(z - e)   = sum_j eps_j xi^j / (r s) T_j,                                eps_0 = 1, eps_j = 2
//   1/(z - e)^2 = sum_j eps_j xi^j [j/s^2 + x/s^3] / r^2 T_j                    (-d/dz)
//   1/(z - e)^3 = sum_j eps_j xi^j [(j^2 - 1)/s^3 + 3 j x/s^4 + 3 x^2/s^5] / (2 r^3) T_j
// The j-independent factors of one frequency:
struct SeriesZ {
  double2 xi, c1, c2a, c2b, c3a, c3b, c3c;  // c1; c2a j + c2b; c3a (j^2 - 1) + c3b j + c3c
};
__device__ __forceinline__ SeriesZ series_z(double dx, double w, double r, bool powers) {
  SeriesZ q;
  const double ir = 1.0 / r;
  const double2 x = make_double2(dx * ir, w * ir);
  // s = sqrt(x^2 - 1) with Im s > 0: from |u| and the larger component first
  const double2 u = make_double2(fma(x.x, x.x, -fma(x.y, x.y, 1.0)), 2.0 * x.x * x.y);
  const double au = sqrt(fma(u.x, u.x, u.y * u.y));
  const double p = sqrt(0.5 * (au + fabs(u.x)));
  const double h = 0.5 * u.y / p;
  double2 s = u.x >= 0.0 ? make_double2(p, h) : make_double2(h, p);
  if (s.y < 0.0 || (s.y == 0.0 && x.x < 0.0)) s = make_double2(-s.x, -s.y);
  q.xi = gj64::crcp_scaled(make_double2(x.x + s.x, x.y + s.y), pivot_key(make_double2(x.x + s.x, x.y + s.y)));
  const double2 is = gj64::crcp_scaled(s, pivot_key(s));
  q.c1 = make_double2(is.x * ir, is.y * ir);
  if (powers) {
    q.c2a = cmul(q.c1, make_double2(is.x * ir, is.y * ir));                  // 1 / (s^2 r^2)
    const double2 t = cmul(x, is);                                           // x / s
    q.c2b = cmul(q.c2a, t);                                                  // x / (s^3 r^2)
    const double g = 0.5 * ir;
    const double2 is2 = make_double2(is.x * g, is.y * g);
    q.c3a = cmul(q.c2a, is2);                                                // 1 / (2 s^3 r^3)
    q.c3b = cmul(q.c2b, make_double2(3.0 * is2.x, 3.0 * is2.y));             // 3 x / (2 s^4 r^3)
    q.c3c = cmul(q.c3b, t);                                                  // 3 x^2 / (2 s^5 r^3)
  }
  return q;
}
// b^j, j < 2^BITS
template <int BITS>
__device__ __forceinline__ double2 cpow_int(double2 b, int j) {
  double2 v = make_double2(1.0, 0.0);
#pragma unroll
  for (int t = 0; t < BITS; ++t) {
    if ((j >> t) & 1) v = cmul(v, b);
    b = cmul(b, b);
  }
  return v;
}

}  // namespace series
}  // namespace gf
