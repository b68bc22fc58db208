// Hankel functions of a far or near point pair below the expansion range
// (x = k R < 24) from per-run tables, for the mixed form's assembly.
//
// Both wavenumbers of a point pair, k and k~ = k (1 + i t), are functions of the
// real x alone once t is fixed, so a run tabulates them:
//   x < 3 : the ascending series of J0, J1, Y0, Y1 (DLMF 10.8) as polynomials in
//           x^2, real for k and complex for k~ (coefficients (1 + i t)^2m), with
//           log x kept apart; HT_M terms leave less than 1e-16;
//   x >= 3: polynomials of degree HT_D - 1 on intervals of length 1/2, interpolated
//           at Chebyshev nodes (the nearest singularity, x = 0, is at least 13
//           half-widths away: the error falls like 26^-12 < 1e-16).
// An evaluation is ~100 FP64 operations without data-dependent loops; the
// backward recurrence and Taylor shift it replaces (hankel01_pair) took ~1500,
// with the lanes of a warp in different branches.
#pragma once
#include "hankel.cuh"

namespace wcs {

constexpr int HT_M = 15;                 // series terms
constexpr int HT_D = 12;                 // polynomial coefficients
constexpr double HT_X0 = 3.0;
constexpr int HT_N = 42;                 // intervals of 1/2 from x = 3 to 24
constexpr double HT_X1 = HT_X0 + 0.5 * HT_N;
constexpr int HT_SERIES = HT_M * 12;     // per term: J0, J1, S0, T1 of k (4), of k~ (4 complex)
constexpr int HT_SIZE = HT_SERIES + 4 + HT_N * HT_D * 8;   // doubles: series, log(1 + i t) and 1 / (1 + i t), intervals

struct HankelTabArgs {
  double t = 0.0;
  double series[HT_SERIES];
  double tail[4];
  double node[HT_D];                     // Chebyshev nodes on [-1, 1]
  double conv[HT_D * HT_D];              // values at the nodes -> monomial coefficients (row: power)
};
// Host: everything of the table that needs no Bessel functions.
void hankel_tab_args(double t, HankelTabArgs& a);

// H0, H1 at k R and k~ R, x = k R in [HT_X0, HT_X1)
__device__ __forceinline__ void hankel_tab_poly(const double* __restrict__ T, double x, zd& H0, zd& H1, zd& G0, zd& G1) {
  const int i = min(HT_N - 1, (int)((x - HT_X0) * 2.0));
  const double u = 4.0 * (x - (HT_X0 + 0.25 + 0.5 * i));
  const double2* c = (const double2*)(T + HT_SERIES + 4 + (int64_t)i * HT_D * 8);
  double2 a = c[4 * (HT_D - 1)], b = c[4 * (HT_D - 1) + 1], d = c[4 * (HT_D - 1) + 2], e = c[4 * (HT_D - 1) + 3];
#pragma unroll
  for (int m = HT_D - 2; m >= 0; --m) {
    const double2 a1 = c[4 * m], b1 = c[4 * m + 1], d1 = c[4 * m + 2], e1 = c[4 * m + 3];
    a.x = fma(a.x, u, a1.x); a.y = fma(a.y, u, a1.y);
    b.x = fma(b.x, u, b1.x); b.y = fma(b.y, u, b1.y);
    d.x = fma(d.x, u, d1.x); d.y = fma(d.y, u, d1.y);
    e.x = fma(e.x, u, e1.x); e.y = fma(e.y, u, e1.y);
  }
  H0 = mkz(a.x, a.y);
  H1 = mkz(b.x, b.y);
  G0 = mkz(d.x, d.y);
  G1 = mkz(e.x, e.y);
}

// The same with J0, J1 of both for x < HT_X0 (lx = log(x / 2))
__device__ __forceinline__ void hankel_tab_series(const double* __restrict__ T, double x, double lx, Hankel01& hk,
                                                  Hankel01& ht) {
  const double X = x * x;
  const double* c = T + (HT_M - 1) * 12;
  double j0 = c[0], j1 = c[1], s0 = c[2], t1 = c[3];
  zd J0 = mkz(c[4], c[5]), J1 = mkz(c[6], c[7]), S0 = mkz(c[8], c[9]), T1 = mkz(c[10], c[11]);
#pragma unroll 2
  for (int m = HT_M - 2; m >= 0; --m) {
    c -= 12;
    j0 = fma(j0, X, c[0]);
    j1 = fma(j1, X, c[1]);
    s0 = fma(s0, X, c[2]);
    t1 = fma(t1, X, c[3]);
    J0 = mkz(fma(J0.x, X, c[4]), fma(J0.y, X, c[5]));
    J1 = mkz(fma(J1.x, X, c[6]), fma(J1.y, X, c[7]));
    S0 = mkz(fma(S0.x, X, c[8]), fma(S0.y, X, c[9]));
    T1 = mkz(fma(T1.x, X, c[10]), fma(T1.y, X, c[11]));
  }
  const double* tail = T + HT_SERIES;
  const double g = 2.0 / WCS_PI, ix = 1.0 / x;
  j1 *= x;
  t1 *= x;
  J1 = x * J1;
  T1 = x * T1;
  // Y0 = (2 / pi) ((log(z / 2) + gamma) J0 + S0), Y1 = (2 / pi) (log(z / 2) J1 - 1 / z) - T1 / pi
  const double y0 = g * fma(lx + WCS_EULER_GAMMA, j0, s0), y1 = fma(g, fma(lx, j1, -ix), -(0.5 * g) * t1);
  const zd lz = mkz(lx + tail[0], tail[1]);
  const zd Y0 = g * ((lz + mkz(WCS_EULER_GAMMA)) * J0 + S0);
  const zd Y1 = g * (lz * J1 - ix * mkz(tail[2], tail[3])) - (0.5 * g) * T1;
  hk.J0 = mkz(j0);
  hk.J1 = mkz(j1);
  hk.H0 = mkz(j0, y0);
  hk.H1 = mkz(j1, y1);
  ht.J0 = J0;
  ht.J1 = J1;
  ht.H0 = mkz(J0.x - Y0.y, J0.y + Y0.x);
  ht.H1 = mkz(J1.x - Y1.y, J1.y + Y1.x);
}

}  // namespace wcs
