// Far element pairs of the mixed form on the FP32 pipe, to the accuracy of the
// stored split-bf16 entries (~1e-9 relative).
//
// GB300's FP64 pipe runs at 1/64 of the FP32 rate, and an entry needs 16 point
// pairs of two Hankel orders at two wavenumbers.  What makes FP32 enough is to
// give it small quantities only.  With element centres c_e, c_f (curve points),
// d0 = c_e - c_f, R0 = |d0|, and the point offsets o_p = r_p - c_e, o_r likewise:
//
//   K(R_pr) = K(R0) Z_p conj(Z_r) (1 + g_pr),
//
// * K(R0): one evaluation per element pair and kernel in float-float (phase,
//   amplitude, damping; the Hankel series is 1 + a term below 1/160);
// * Z_p = e^{i alpha_e s_p}, alpha_e = k h (d0 . tau_e) / R0, s_p = xi_p - 1/2:
//   the part of the phase that is linear along the tangents.  Its weighted sum
//   over an element is a function of alpha alone, A_0 = conj(A_1) =
//   sum_p w_p phi_0(xi_p) e^{i alpha s_p} = 1/2 - i alpha / 12 + O(alpha^2) (a
//   polynomial with per-run coefficients), so the sum over both elements is the
//   exact 1/4, a float-float term linear in alpha, and a small remainder;
// * g_pr: what curvature and the second-order distance add, (1 + rho)^-1/2 for
//   the amplitude, e^{-Im k~ (R - R0)}, and the change of the Hankel series: a
//   few hundredths at k R0 = 20 and less beyond, summed over the point pairs in
//   FP32.
//
// The double-layer factor (r - r').n' / R and the Maue factor n.n' are split the
// same way into their value at the centres (float-float) and a small deviation.
//
// FP32 roundings therefore enter at 1e-2 of the entry: 3e-9 (N) to 7e-9 (D) of it
// rms at k h = 0.63 against FP64 quadrature of the same points, 2^-24.7 of the kernel at
// worst up to k h = 0.9 and elements that turn by a radian (the CPU build of
// tests/test_far_pairs_cpu.py and test_far_pairs_curved_cpu.py), and the solution errors against 64-bit references
// are those of FP64 integration.  Bound: FP32 issue, ~3300 instructions a pair.
#pragma once
#include "common.cuh"

namespace wcs {

#define WCS_HD __host__ __device__ __forceinline__

struct cf {
  float x, y;
};
WCS_HD cf cmul(cf a, cf b) { return {fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x)}; }
// a * conj(b)
WCS_HD cf cmulc(cf a, cf b) { return {fmaf(a.x, b.x, a.y * b.y), fmaf(a.y, b.x, -a.x * b.y)}; }
WCS_HD cf cfma(cf a, cf b, cf c) {   // a b + c
  return {fmaf(a.x, b.x, fmaf(-a.y, b.y, c.x)), fmaf(a.x, b.y, fmaf(a.y, b.x, c.y))};
}
WCS_HD void caxpy(cf& acc, float s, cf v) {
  acc.x = fmaf(s, v.x, acc.x);
  acc.y = fmaf(s, v.y, acc.y);
}

// Float-float arithmetic (value = hi + lo, ~48 bits; Dekker/Knuth error-free
// transformations), on the FP32 pipe.
struct ff {
  float hi, lo;
};
WCS_HD ff ff_quick(float a, float b) {
  const float s = a + b;
  return {s, b - (s - a)};
}
WCS_HD ff ff_two_sum(float a, float b) {
  const float s = a + b;
  const float bb = s - a;
  return {s, (a - (s - bb)) + (b - bb)};
}
WCS_HD ff ff_two_prod(float a, float b) {
  const float p = a * b;
  return {p, fmaf(a, b, -p)};
}
WCS_HD ff ff_add(ff a, ff b) {
  const ff s = ff_two_sum(a.hi, b.hi);
  return ff_quick(s.hi, s.lo + (a.lo + b.lo));
}
WCS_HD ff ff_add_f(ff a, float b) {
  const ff s = ff_two_sum(a.hi, b);
  return ff_quick(s.hi, s.lo + a.lo);
}
WCS_HD ff ff_neg(ff a) { return {-a.hi, -a.lo}; }
WCS_HD ff ff_mul(ff a, ff b) {
  ff p = ff_two_prod(a.hi, b.hi);
  return ff_quick(p.hi, p.lo + fmaf(a.hi, b.lo, a.lo * b.hi));
}
WCS_HD ff ff_of(double x) {
  const float h = (float)x;
  return ff{h, (float)(x - (double)h)};
}
// 1 / x for a factor of the small corrections (2 ulp)
WCS_HD float far_rcp(float x) {
#ifdef __CUDA_ARCH__
  return __fdividef(1.f, x);
#else
  return 1.f / x;
#endif
}
// FP32 seeds of the Newton steps below (their error is squared away)
WCS_HD float ff_seed_rsqrt(float x) {
#ifdef __CUDA_ARCH__
  return rsqrtf(x);
#else
  return 1.f / sqrtf(x);
#endif
}
// x^-1/2
WCS_HD ff ff_rsqrt(ff x) {
  const float y = ff_seed_rsqrt(x.hi);
  // 1 - x y^2, a small number
  const ff y2 = ff_two_prod(y, y);
  const ff p = ff_mul(x, y2);
  const float e = (1.f - p.hi) - p.lo;
  return ff_quick(y, y * (0.5f * e) * fmaf(0.75f, e, 1.f));
}

// sin and cos of a float-float angle, |x| <= 4
WCS_HD void ff_sincos(ff x, ff& s, ff& c) {
  const float j = rintf(x.hi * 0.636619747f);
  // pi / 2 = 1.57079637 - 4.37113883e-8 - 1.71512489e-15
  ff r = ff_add(x, ff_neg(ff_two_prod(j, 1.57079637f)));
  r = ff_add_f(r, j * 4.37113883e-08f);
  const ff z = ff_mul(r, r);
  // cos r = 1 - z / 2 + z^2 (1/24 - z / 720 + ...)
  const float zz = z.hi;
  const float tc = zz * zz * fmaf(zz, fmaf(zz, fmaf(zz, -2.75573188e-07f, 2.48015876e-05f), -1.38888892e-03f), 4.16666679e-02f);
  ff cc = ff_two_sum(1.f, -0.5f * z.hi);
  cc = ff_quick(cc.hi, cc.lo + (tc - 0.5f * z.lo));
  // sin r = r - r z / 6 + r z^2 (1/120 - z / 5040 + ...)
  const ff rz = ff_mul(ff_mul(r, z), ff{-0.16666667f, 4.96705388e-09f});
  const float ts = r.hi * zz * zz * fmaf(zz, fmaf(zz, 2.75573188e-06f, -1.98412701e-04f), 8.33333377e-03f);
  ff ss = ff_add(r, rz);
  ss = ff_quick(ss.hi, ss.lo + ts);
  const int q = ((int)j) & 3;
  const bool sw = q & 1;
  const ff a = sw ? cc : ss, b = sw ? ss : cc;
  s = (q & 2) ? ff_neg(a) : a;
  c = (q == 1 || q == 2) ? ff_neg(b) : b;
}

// e^-x for a float-float x >= 0 (zero beyond the FP32 range)
WCS_HD ff ff_exp_neg(ff x) {
  const float n = rintf(x.hi * 1.44269502f);
  // ln 2 = 0.693147182 - 1.90465421e-9
  ff r = ff_add(x, ff_neg(ff_two_prod(n, 0.693147182f)));
  r = ff_add_f(r, n * 1.90465421e-09f);
  const float v = r.hi;
  const ff h = ff_two_prod(v, v);
  float t3 = fmaf(v, fmaf(v, 2.75573188e-06f, -2.48015876e-05f), 1.98412701e-04f);
  t3 = v * h.hi * fmaf(v, fmaf(v, fmaf(v, fmaf(v, t3, -1.38888892e-03f), 8.33333377e-03f), -4.16666679e-02f), 0.166666672f);
  // 1 - r + r^2 / 2 - (r^3 / 6 - ...)
  ff y = ff_two_sum(1.f, -r.hi);
  y = ff_add(y, ff{0.5f * h.hi, 0.5f * h.lo});
  y = ff_quick(y.hi, y.lo + (fmaf(r.lo, r.hi - 1.f, 0.f) - t3));
  if (n > 120.f) return {0.f, 0.f};
#ifdef __CUDA_ARCH__
  const float sc = __int_as_float((127 - (int)n) << 23);
#else
  const float sc = ldexpf(1.f, -(int)n);
#endif
  return {y.hi * sc, y.lo * sc};
}

// Per-run constants of the far pairs, formed on the host and passed by value.
constexpr int FAR_Q = 16;      // most points per element
constexpr int FAR_P = 6;       // terms of the tangential polynomials
constexpr int FAR_M = 8;       // terms of the Hankel series (k R >= 20: the first omitted one is below 3e-10)
struct FarConsts {
  float xmin2 = 0.f;               // smallest k^2 R0^2 of the route
  ff k{0.f, 0.f}, kh{0.f, 0.f}, beta{0.f, 0.f};   // k, k h, Im k~
  float ikt[2] = {0.f, 0.f};       // 1 / (1 + i t), k~ = k (1 + i t)
  ff kk2h2{0.f, 0.f};              // k^2 h^2 of the Maue form
  float hf = 0.f;                  // h
  float w[2][FAR_Q] = {}, w1[FAR_Q] = {}, s[FAR_Q] = {};   // w_p phi_a(xi_p), w_p, xi_p - 1/2
  float pe[FAR_P] = {}, po[FAR_P] = {};    // Re A_0 - 1/2 = sum pe_m alpha^2(m+1); Im A_0 + alpha / 12 = alpha sum po_m alpha^2(m+1)
  float a[2][FAR_M] = {};          // a_m(nu) of the Hankel expansion
};

// Per element: centre and tangent as float-float (n = (tau_y, -tau_x)).
struct FarElem {
  float4 c;    // x hi, x lo, y hi, y lo
  float4 t;    // tau_x hi, lo, tau_y hi, lo
};
// Per point: a = offset from the centre (x, y) and its curved part o - h s tau (x, y);
// b = deviation of the normal from the centre's (x, y), o . tau, o . n; c = o . n(point)
struct FarPoint {
  float4 a, b;
  float c, o2, pad0, pad1;     // o2 = |o|^2
};

// Table entries from FP64 geometry: (cx, cy) the centre, (nx, ny) its normal;
// (x, y), (px, py) a point and its normal at s = xi - 1/2.
WCS_HD FarElem far_elem(double cx, double cy, double nx, double ny) {
  const ff x = ff_of(cx), y = ff_of(cy), tx = ff_of(-ny), ty = ff_of(nx);
  FarElem e;
  e.c.x = x.hi; e.c.y = x.lo; e.c.z = y.hi; e.c.w = y.lo;
  e.t.x = tx.hi; e.t.y = tx.lo; e.t.z = ty.hi; e.t.w = ty.lo;
  return e;
}
WCS_HD FarPoint far_point(double cx, double cy, double nx, double ny, double x, double y, double px, double py, double h,
                          double s) {
  const double ox = x - cx, oy = y - cy, tx = -ny, ty = nx;
  FarPoint p;
  p.a.x = (float)ox; p.a.y = (float)oy;
  p.a.z = (float)(ox - h * s * tx); p.a.w = (float)(oy - h * s * ty);
  p.b.x = (float)(px - nx); p.b.y = (float)(py - ny);
  p.b.z = (float)(ox * tx + oy * ty); p.b.w = (float)(ox * nx + oy * ny);
  p.c = (float)(ox * px + oy * py);
  p.o2 = (float)(ox * ox + oy * oy);
  p.pad0 = p.pad1 = 0.f;
  return p;
}

// Constants of a run: rule (q nodes xi, weights w on [0, 1]), k, Im k~, h; pairs with k R0 >= xmin.
inline void far_consts(FarConsts& F, int q, const double* xi, const double* w, double k, double beta, double h,
                       double xmin) {
  F = FarConsts{};
  F.xmin2 = (xmin < 1e18) ? (float)(xmin * xmin) : INFINITY;
  F.k = ff_of(k);
  F.kh = ff_of(k * h);
  F.beta = ff_of(beta);
  const double t = beta / k, d = 1.0 + t * t;
  F.ikt[0] = (float)(1.0 / d);
  F.ikt[1] = (float)(-t / d);
  F.kk2h2 = ff_of(k * k * h * h);
  F.hf = (float)h;
  double me[2 * FAR_P + 2] = {};    // moments sum_p w_p (1 - xi_p) s_p^m
  for (int p = 0; p < q; ++p) {
    const double s = xi[p] - 0.5;
    F.s[p] = (float)s;
    F.w[0][p] = (float)(w[p] * (1.0 - xi[p]));
    F.w[1][p] = (float)(w[p] * xi[p]);
    F.w1[p] = (float)w[p];
    double m = w[p] * (1.0 - xi[p]);
    for (int j = 0; j < 2 * FAR_P + 2; ++j) { me[j] += m; m *= s; }
  }
  double fact = 1.0, sg = -1.0;
  for (int m = 0; m < FAR_P; ++m) {
    // alpha^2(m+1): even moment 2m + 2, odd moment 2m + 3
    fact *= (2.0 * m + 1.0) * (2.0 * m + 2.0);
    F.pe[m] = (float)(sg * me[2 * m + 2] / fact);
    F.po[m] = (2 * m + 3 < 2 * FAR_P + 2) ? (float)(sg * me[2 * m + 3] / (fact * (2.0 * m + 3.0))) : 0.f;
    sg = -sg;
  }
  for (int nu = 0; nu < 2; ++nu) {
    double a = 1.0;
    for (int m = 0; m < FAR_M; ++m) {
      if (m > 0) a *= (4.0 * nu * nu - (2.0 * m - 1.0) * (2.0 * m - 1.0)) / (8.0 * m);
      F.a[nu][m] = (float)a;
    }
  }
}

struct ffc {
  ff x, y;
};
WCS_HD ffc ffc_mul(ffc a, ff s) { return {ff_mul(a.x, s), ff_mul(a.y, s)}; }

// One element pair (e, f): the reference kernels, the exact leading parts and the
// FP32 corrections of the operators, [a * 2 + b] (a: hat on e, b: hat on f).  With
// the factors fS = (i/4) sqrt(2 / (pi k~)) h^2, fD = (i/4) sqrt(2 / (pi k)) k h^2,
// fDt = fS k~ and fN = (i/4) sqrt(2 / (pi k)) an integral is f (lead + K (i lam +
// corr)) (see value()).  M: also D and D~ of the mirrored pair (f, e) (operators 4
// and 5); its S~ and N are this pair's, and every Hankel evaluation is shared.
template <bool M>
struct FarPair {
  static constexpr int OPS = M ? 6 : 4;
  ffc lead[OPS + 1];           // S~, D, D~ (a quarter of the kernel), N for a = b, [D, D~ mirrored,] N for a != b
  cf K[OPS];                   // T0, K1 g, T1 g, -, K1 g', T1 g' (heads): factors of the linear phase term
  ff lam[2];                   // (alpha_e - alpha_f) / 24 for a = b = 0, (alpha_e + alpha_f) / 24 for a = 0, b = 1
  cf corr[OPS][4];             // K times the corrections

  WCS_HD ffc value(int op, int j) const {
    const ffc& l = lead[(op == 3 && (j == 1 || j == 2)) ? OPS : op];
    const cf c = corr[op][j];
    ff x = ff_two_sum(l.x.hi, c.x), y = ff_two_sum(l.y.hi, c.y);
    x.lo += l.x.lo;
    y.lo += l.y.lo;
    if (op != 3) {
      // K (i lam): (-K.y lam, K.x lam) with the rounding errors of the products
      const ff la = lam[(j == 1 || j == 2) ? 1 : 0];
      const float sg = (j >= 2) ? -1.f : 1.f;    // j = 2, 3 mirror j = 1, 0
      const float lh = -sg * la.hi;               // Im A_0 = -alpha / 12
      const ff px = ff_two_prod(-K[op].y, lh), py = ff_two_prod(K[op].x, lh);
      const ff sx = ff_two_sum(x.hi, px.hi), sy = ff_two_sum(y.hi, py.hi);
      x = {sx.hi, sx.lo + (x.lo + fmaf(K[op].y, sg * la.lo, px.lo))};
      y = {sy.hi, sy.lo + (y.lo + fmaf(-K[op].x, sg * la.lo, py.lo))};
    }
    return {x, y};
  }
};

WCS_HD bool far_ok(const FarConsts& F, const float4& ce, const float4& cg) {
  const float dx = ce.x - cg.x, dy = ce.z - cg.z;
  return F.k.hi * F.k.hi * (dx * dx + dy * dy) >= F.xmin2;
}

// Hankel series at w = i u, u = 1 / (k R0) (or 1 / (k~ R0)): s = sum_{m>=1} a_m w^m,
// and the coefficients b1, b2 of its change with v = R0 / R - 1 relative to
// 1 + s: b1 v + b2 v^2.
WCS_HD cf far_recip1(cf s) {   // 1 / (1 + s)
  const float x = 1.f + s.x, iq = 1.f / fmaf(x, x, s.y * s.y);
  return {x * iq, -s.y * iq};
}
WCS_HD void far_series(const float* a, float u, cf& s, cf& b1, cf& b2) {
  // even and odd powers of w = i u: real polynomials in -u^2
  const float z = -u * u;
  float se = a[6], so = a[7], de = 6.f * a[6], od = 7.f * a[7], ee = 15.f * a[6], eo = 10.f * a[5];
  se = fmaf(se, z, a[4]);
  so = fmaf(so, z, a[5]);
  de = fmaf(de, z, 4.f * a[4]);
  od = fmaf(od, z, 5.f * a[5]);
  ee = fmaf(ee, z, 6.f * a[4]);
  eo = fmaf(eo, z, 3.f * a[3]);
  se = fmaf(se, z, a[2]);
  so = fmaf(so, z, a[3]);
  de = fmaf(de, z, 2.f * a[2]);
  od = fmaf(od, z, 3.f * a[3]);
  ee = fmaf(ee, z, a[2]);
  so = fmaf(so, z, a[1]);
  od = fmaf(od, z, a[1]);
  s = {se * z, so * u};
  const cf r = far_recip1(s);
  b1 = cmul({de * z, od * u}, r);
  b2 = cmul({ee * z, eo * u * z}, r);
}
WCS_HD void far_series_c(const float* a, cf w, cf& s, cf& b1) {
  cf p = {a[FAR_M - 1], 0.f}, d = {(FAR_M - 1) * a[FAR_M - 1], 0.f};
#pragma unroll
  for (int m = FAR_M - 2; m >= 1; --m) {
    p = cmul(p, w);
    p.x += a[m];
    d = cmul(d, w);
    d.x += m * a[m];
  }
  s = cmul(p, w);
  b1 = cmul(cmul(d, w), far_recip1(s));
}

// e^{i x}, |x| <= 1.2 (k h <= 2.5, |s| < 1/2), to the FP32 accuracy the corrections need
WCS_HD void far_cis(float x, cf& z) {
  const float x2 = x * x;
  z.y = fmaf(x * x2, fmaf(x2, fmaf(x2, fmaf(x2, 2.75573188e-06f, -1.98412701e-04f), 8.33333377e-03f), -0.166666672f), x);
  z.x = fmaf(x2, fmaf(x2, fmaf(x2, fmaf(x2, 2.48015876e-05f, -1.38888892e-03f), 4.16666679e-02f), -0.5f), 1.f);
}

// K + K s, s a small complex number
WCS_HD ffc ffc_grow(const ffc& K, cf s) {
  const float px = fmaf(K.x.hi, s.x, -K.y.hi * s.y), py = fmaf(K.x.hi, s.y, K.y.hi * s.x);
  return {ff_add_f(K.x, px), ff_add_f(K.y, py)};
}

template <int Q, bool M>   // points per element (0: q at run time); mirrored pair as well
WCS_HD void far_pair(const FarConsts& F, int q_run, const FarElem& E, const FarElem& G, const FarPoint* pe,
                     const FarPoint* pg, FarPair<M>& o) {
  const int q = Q ? Q : q_run;
  // ---- geometry of the centres
  const ff dx = ff_add(ff_two_sum(E.c.x, -G.c.x), ff_two_sum(E.c.y, -G.c.y));
  const ff dy = ff_add(ff_two_sum(E.c.z, -G.c.z), ff_two_sum(E.c.w, -G.c.w));
  const ff R02 = ff_add(ff_mul(dx, dx), ff_mul(dy, dy));
  const ff iR0 = ff_rsqrt(R02);
  const ff R0 = ff_mul(R02, iR0);
  const ff kR0 = ff_mul(F.k, R0);
  const float ir = iR0.hi, kr = kR0.hi, ir2 = ir * ir;
  const ff tex = {E.t.x, E.t.y}, tey = {E.t.z, E.t.w}, tgx = {G.t.x, G.t.y}, tgy = {G.t.z, G.t.w};
  const ff khr = ff_mul(F.kh, iR0);
  const ff ae = ff_mul(khr, ff_add(ff_mul(dx, tex), ff_mul(dy, tey)));
  const ff ag = ff_mul(khr, ff_add(ff_mul(dx, tgx), ff_mul(dy, tgy)));
  // n = (tau_y, -tau_x): (c_e - c_f) . n_f / R0, n_e . n_f = tau_e . tau_f, tau_e . n_f
  const ff g0 = ff_mul(iR0, ff_add(ff_mul(dx, tgy), ff_neg(ff_mul(dy, tgx))));
  const ff nd0 = ff_add(ff_mul(tex, tgx), ff_mul(tey, tgy));
  const ff sg_ff = ff_add(ff_mul(tex, tgy), ff_neg(ff_mul(tey, tgx)));
  const float sg = sg_ff.hi, ndh = nd0.hi, g0h = g0.hi;
  // mirrored pair: (c_f - c_e) . n_e / R0 (n_e = (tau_y, -tau_x))
  ff gm = {0.f, 0.f};
  if (M) gm = ff_mul(iR0, ff_add(ff_mul(dy, tex), ff_neg(ff_mul(dx, tey))));
  const float gmh = gm.hi;
  const float dxh = dx.hi, dyh = dy.hi, ux = dxh * ir, uy = dyh * ir;
  // ---- reference kernels
  // k R0 - n 2 pi, 2 pi = 6.28318548 - 1.74845553e-7 - 6.86049999e-15 (n < 2^13), less pi / 4
  const float n = rintf(kr * 0.15915494f);
  ff ph = ff_add(kR0, ff_neg(ff_two_prod(n, 6.28318548f)));
  ph = ff_add(ph, ff_two_prod(n, 1.74845553e-07f));
  ph = ff_add(ff_add_f(ph, n * 6.86049999e-15f), ff{-0.785398185f, 2.18556941e-08f});
  ff sn, cs;
  ff_sincos(ph, sn, cs);
  const ff am = ff_rsqrt(R0);
  const ffc E1 = {ff_mul(cs, am), ff_mul(sn, am)};
  const ff damp = ff_exp_neg(ff_mul(F.beta, R0));
  const ffc Et = ffc_mul(E1, damp);
  const float u = 1.f / kr;
  const cf wt = {-F.ikt[1] * u, F.ikt[0] * u};
  cf s0, s1, s0t, s1t, b10, b20, b11, b21, b10t, b11t;
  far_series(F.a[0], u, s0, b10, b20);
  far_series(F.a[1], u, s1, b11, b21);
  far_series_c(F.a[0], wt, s0t, b10t);
  far_series_c(F.a[1], wt, s1t, b11t);
  // the v^2 terms (4e-7 of the kernel at k R0 = 20) follow those of k through their
  // leading power: b2(k~) = b2(k) (1 + i t)^-2 to ~1e-9 of the kernel
  const cf ik1 = {F.ikt[0], F.ikt[1]}, ik2 = cmul(ik1, ik1);
  const cf b20t = cmul(b20, ik2), b21t = cmul(b21, ik2);
  const ffc K0 = ffc_grow(E1, s0), K1r = ffc_grow(E1, s1), T0 = ffc_grow(Et, s0t), T1r = ffc_grow(Et, s1t);
  const ffc K1 = {K1r.y, {-K1r.x.hi, -K1r.x.lo}}, T1 = {T1r.y, {-T1r.x.hi, -T1r.x.lo}};   // times -i

  // ---- corrections: sums over the point pairs (c0 without hats as well: the
  // derivative part of N)
  cf vS[4], vD[4], vt[4], vN[4], vDm[4], vtm[4], v0 = {0.f, 0.f};
#pragma unroll
  for (int j = 0; j < 4; ++j) vS[j] = vD[j] = vt[j] = vN[j] = vDm[j] = vtm[j] = cf{0.f, 0.f};
  const float aef = ae.hi, agf = ag.hi, hir = F.hf * ir;
  const float bR = F.beta.hi * R0.hi;
  const float lte = hir * fmaf(dxh, tex.hi, dyh * tey.hi), ltg = hir * fmaf(dxh, tgx.hi, dyh * tgy.hi);
  // source points: phase factor, tangential and curved displacement along d0, d0 . nu_r - o_r . n_r
  constexpr int QR = Q ? Q : 1;
  cf Zr_[QR];
  float tr_[QR], er_[QR], Kr_[QR];
  auto source = [&](int r, cf& Zr, float& tr, float& er, float& Kr) {
    const float4 ra = pg[r].a;
    far_cis(agf * F.s[r], Zr);
    er = fmaf(ux, ra.z, uy * ra.w);
    tr = fmaf(ltg, F.s[r], er);
    Kr = fmaf(dxh, pg[r].b.x, dyh * pg[r].b.y) - pg[r].c;
  };
  if (Q) {
#pragma unroll
    for (int r = 0; r < QR; ++r) source(r, Zr_[r], tr_[r], er_[r], Kr_[r]);
  }
#pragma unroll 1
  for (int p = 0; p < q; ++p) {
    const float4 pa = pe[p].a, pb = pe[p].b;
    const float po2 = pe[p].o2;
    cf Zp;
    far_cis(aef * F.s[p], Zp);
    const float ep = fmaf(ux, pa.z, uy * pa.w);        // d0 . (curved part) / R0
    const float tp = fmaf(lte, F.s[p], ep);
    const float Lp = fmaf(pb.z, sg, pb.w * ndh);       // o_p . n_f
    const float np = fmaf(pb.x, tgy.hi, -pb.y * tgx.hi);
    const float Kp = -fmaf(dxh, pb.x, dyh * pb.y) - pe[p].c;   // mirrored: -d0 . nu_p - o_p . n_p
    cf uS[2], uD[2], ut[2], uN[2], uDm[2], utm[2], u0 = {0.f, 0.f};
#pragma unroll
    for (int b = 0; b < 2; ++b) uS[b] = uD[b] = ut[b] = uN[b] = uDm[b] = utm[b] = cf{0.f, 0.f};
#pragma unroll
    for (int r = 0; r < (Q ? Q : FAR_Q); ++r) {
      if (!Q && r >= q) break;
      const float4 ra = pg[r].a, rb = pg[r].b;
      cf Zr;
      float tr, er, Kr;
      if (Q) {
        Zr = Zr_[r < QR ? r : 0];
        tr = tr_[r < QR ? r : 0];
        er = er_[r < QR ? r : 0];
        Kr = Kr_[r < QR ? r : 0];
      } else {
        source(r, Zr, tr, er, Kr);
      }
      // rho = R / R0 - 1 = tau + x-terms, tau = d0.D / R0^2, D = o_p - o_r
      const float tau = (tp - tr) * ir;
      const float d2 = (fmaf(-2.f, fmaf(pa.x, ra.x, pa.y * ra.y), po2 + pg[r].o2)) * ir2;
      const float nu = fmaf(-tau, tau, d2);
      const float o1 = 1.f + tau, io = far_rcp(o1);
      const float x = nu * io * io;
      const float sec = o1 * x * fmaf(x, fmaf(x, 0.0625f, -0.125f), 0.5f);
      const float rho = tau + sec;
      // phase beyond the tangential part
      const float eta = fmaf(kr, sec, F.k.hi * (ep - er));
      const float e2 = eta * eta;
      const cf ei = {e2 * fmaf(e2, fmaf(e2, -1.38888892e-03f, 4.16666679e-02f), -0.5f),
                     fmaf(eta * e2, fmaf(e2, 8.33333377e-03f, -0.166666672f), eta)};
      // (1 + rho)^-1/2 - 1 and R0 / R - 1
      const float am1 = rho * fmaf(rho, fmaf(rho, fmaf(rho, fmaf(rho, fmaf(rho, 0.225585938f, -0.24609375f), 0.2734375f),
                                                       -0.3125f), 0.375f), -0.5f);
      const float v = fmaf(am1, am1, am1 + am1);
      const float y = bR * rho;
      const float dm1 = y * fmaf(y, fmaf(y, fmaf(y, 4.16666679e-02f, -0.166666672f), 0.5f), -1.f);
      const float at = fmaf(am1, dm1, am1 + dm1);
      const cf gk = {fmaf(am1, ei.x, ei.x + am1), fmaf(am1, ei.y, ei.y)};
      const cf gt = {fmaf(at, ei.x, ei.x + at), fmaf(at, ei.y, ei.y)};
      const cf Z = cmulc(Zp, Zr);
      const cf Ck = cmul(Z, gk), Ct = cmul(Z, gt);
      const cf Pk = {Z.x + Ck.x, Z.y + Ck.y}, Pt = {Z.x + Ct.x, Z.y + Ct.y};
      const cf q0 = {v * fmaf(v, b20.x, b10.x), v * fmaf(v, b20.y, b10.y)};
      const cf q1 = {v * fmaf(v, b21.x, b11.x), v * fmaf(v, b21.y, b11.y)};
      const cf q0t = {v * fmaf(v, b20t.x, b10t.x), v * fmaf(v, b20t.y, b10t.y)};
      const cf q1t = {v * fmaf(v, b21t.x, b11t.x), v * fmaf(v, b21t.y, b11t.y)};
      // (r - r').n' / R = g0 + gd: (d0.nu_r + o_p.n_f + o_p.nu_r - o_r.n_r) / R0 - g0 rho, over 1 + rho
      const float sr = Kr + fmaf(pa.x, rb.x, fmaf(pa.y, rb.y, Lp));
      const float gd = fmaf(sr, ir, -g0h * rho) * (1.f + v);
      // n_p . n_r = nd0 + nn
      const float nn = np + fmaf(tey.hi, rb.x, fmaf(-tex.hi, rb.y, fmaf(pb.x, rb.x, pb.y * rb.y)));
      // per function: c = C + q P (the kernel's deviation), then f0 c + fd (P + q P) = (f0 + fd) c + fd Z with
      // f0, fd the factor at the centres and its deviation
      const cf c0 = cfma(q0, Pk, Ck), c1 = cfma(q1, Pk, Ck), cS = cfma(q0t, Pt, Ct), ct = cfma(q1t, Pt, Ct);
      const float gs = g0h + gd, ns = ndh + nn;
      const cf yD = {fmaf(gs, c1.x, gd * Z.x), fmaf(gs, c1.y, gd * Z.y)};
      const cf yt = {fmaf(gs, ct.x, gd * Z.x), fmaf(gs, ct.y, gd * Z.y)};
      const cf yN = {fmaf(ns, c0.x, nn * Z.x), fmaf(ns, c0.y, nn * Z.y)};
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const float wr = F.w[b][r];
        caxpy(uS[b], wr, cS);
        caxpy(uD[b], wr, yD);
        caxpy(ut[b], wr, yt);
        caxpy(uN[b], wr, yN);
      }
      if (M) {
        // o_r . n_p = o_r . n_e + o_r . nu_p, tau_f . n_e = -tau_e . n_f
        const float sm = Kp + fmaf(ra.x, pb.x, fmaf(ra.y, pb.y, fmaf(-rb.z, sg, rb.w * ndh)));
        const float gdm = fmaf(sm, ir, -gmh * rho) * (1.f + v), gsm = gmh + gdm;
        const cf ym = {fmaf(gsm, c1.x, gdm * Z.x), fmaf(gsm, c1.y, gdm * Z.y)};
        const cf yn = {fmaf(gsm, ct.x, gdm * Z.x), fmaf(gsm, ct.y, gdm * Z.y)};
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          caxpy(uDm[b], F.w[b][r], ym);
          caxpy(utm[b], F.w[b][r], yn);
        }
      }
      caxpy(u0, F.w1[r], c0);
    }
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      const float wp = F.w[a][p];
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        caxpy(vS[a * 2 + b], wp, uS[b]);
        caxpy(vD[a * 2 + b], wp, uD[b]);
        caxpy(vt[a * 2 + b], wp, ut[b]);
        caxpy(vN[a * 2 + b], wp, uN[b]);
        if (M) {
          caxpy(vDm[a * 2 + b], wp, uDm[b]);
          caxpy(vtm[a * 2 + b], wp, utm[b]);
        }
      }
    }
    caxpy(v0, F.w1[p], u0);
  }
  // ---- tangential sums: A_0(alpha) = 1/2 + re + i (-alpha / 12 + im), A_1 = conj(A_0)
  float ree = 0.f, ime = 0.f, reg = 0.f, img = 0.f;
  {
    const float ze = aef * aef, zg = agf * agf;
    float e1 = F.pe[FAR_P - 1], e2 = F.po[FAR_P - 1], g1 = F.pe[FAR_P - 1], g2 = F.po[FAR_P - 1];
#pragma unroll
    for (int m = FAR_P - 2; m >= 0; --m) {
      e1 = fmaf(e1, ze, F.pe[m]);
      e2 = fmaf(e2, ze, F.po[m]);
      g1 = fmaf(g1, zg, F.pe[m]);
      g2 = fmaf(g2, zg, F.po[m]);
    }
    ree = ze * e1;
    reg = zg * g1;
    ime = aef * ze * e2;
    img = agf * zg * g2;
  }
  const float lie = aef * (-1.f / 12.f) + ime, lig = agf * (-1.f / 12.f) + img;   // Im A_0 in all
  // A_a(alpha_e) conj(A_b(alpha_f)) - 1/4 = i lam_ab + M_ab; lam_ab = (-sa alpha_e + sb alpha_f) / 24 with s_0 = 1, s_1 = -1
  o.lam[0] = ff_mul(ff_add(ae, ff_neg(ag)), ff{0.0416666679f, -1.24176347e-09f});
  o.lam[1] = ff_mul(ff_add(ae, ag), ff{0.0416666679f, -1.24176347e-09f});
  cf T[4];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const float sa = a ? -1.f : 1.f, sb = b ? -1.f : 1.f;
      // x = re_e + i sa lie, y = re_g - i sb lig (conjugated)
      const float xi = sa * lie, yi = -sb * lig;
      T[a * 2 + b] = {fmaf(0.5f, ree + reg, fmaf(ree, reg, -xi * yi)),
                      fmaf(0.5f, fmaf(sa, ime, -sb * img), fmaf(ree, yi, reg * xi))};
    }
  // ---- assemble leads and corrections
  const cf k0 = {K0.x.hi, K0.y.hi}, k1 = {K1.x.hi, K1.y.hi}, t0 = {T0.x.hi, T0.y.hi}, t1 = {T1.x.hi, T1.y.hi};
  const ff q4 = {0.25f, 0.f};
  o.lead[0] = {{0.25f * T0.x.hi, 0.25f * T0.x.lo}, {0.25f * T0.y.hi, 0.25f * T0.y.lo}};
  const ff g4 = {0.25f * g0.hi, 0.25f * g0.lo};
  o.lead[1] = ffc_mul(K1, g4);
  o.lead[2] = ffc_mul(T1, g4);
  // N: +-1 - k^2 h^2 nd0 / 4
  const ff mq = ff_mul(ff_mul(F.kk2h2, nd0), q4);
  o.lead[3] = ffc_mul(K0, ff_add_f(ff_neg(mq), 1.f));
  o.lead[FarPair<M>::OPS] = ffc_mul(K0, ff_add_f(ff_neg(mq), -1.f));
  o.K[0] = t0;
  o.K[1] = {k1.x * g0h, k1.y * g0h};
  o.K[2] = {t1.x * g0h, t1.y * g0h};
  o.K[3] = {0.f, 0.f};
  if (M) {
    const ff m4 = {0.25f * gm.hi, 0.25f * gm.lo};
    o.lead[4] = ffc_mul(K1, m4);
    o.lead[M ? 5 : 0] = ffc_mul(T1, m4);
    o.K[M ? 4 : 0] = {k1.x * gmh, k1.y * gmh};
    o.K[M ? 5 : 0] = {t1.x * gmh, t1.y * gmh};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      o.corr[M ? 4 : 0][j] = cmul(k1, {fmaf(gmh, T[j].x, vDm[j].x), fmaf(gmh, T[j].y, vDm[j].y)});
      o.corr[M ? 5 : 0][j] = cmul(t1, {fmaf(gmh, T[j].x, vtm[j].x), fmaf(gmh, T[j].y, vtm[j].y)});
    }
  }
  cf sum0 = v0;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    sum0.x += T[j].x;
    sum0.y += T[j].y;
  }
  const float kk = F.kk2h2.hi;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    o.corr[0][j] = cmul(t0, {vS[j].x + T[j].x, vS[j].y + T[j].y});
    o.corr[1][j] = cmul(k1, {fmaf(g0h, T[j].x, vD[j].x), fmaf(g0h, T[j].y, vD[j].y)});
    o.corr[2][j] = cmul(t1, {fmaf(g0h, T[j].x, vt[j].x), fmaf(g0h, T[j].y, vt[j].y)});
    const float lm = ((j >= 2) ? 1.f : -1.f) * o.lam[(j == 1 || j == 2) ? 1 : 0].hi;
    const float sgn = (j == 0 || j == 3) ? 1.f : -1.f;
    const cf c0 = {fmaf(ndh, T[j].x, vN[j].x), fmaf(ndh, T[j].y + lm, vN[j].y)};
    o.corr[3][j] = cmul(k0, {fmaf(-kk, c0.x, sgn * sum0.x), fmaf(-kk, c0.y, sgn * sum0.y)});
  }
}

}  // namespace wcs
