// Galerkin assembly of the operators of Eq. (4) and Eq. (5):
//   S~ = <l_i, S^k~ l_j>   kernel g_k~ = (i/4) H0(k~ R)
//   D  = <l_i, D^k  l_j>   kernel dg_k/dn' = (i k/4) H1(k R) (r - r').n' / R
//   D~ = <l_i, D^k~ l_j>
//   N  = <l_i, N^k  l_j>   Maue form: [l_i' l_j' - k^2 (n.n') l_i l_j] g_k
// with piecewise-linear hats on the arc-length-uniform mesh (Sec. V).
//
// Element pair (e, f) contributes a 2x2 block to node pairs (e+a, f+b).  One
// CTA owns a 32 x 32 tile of node pairs and evaluates the 33 x 33 element
// pairs that touch it (one Hankel evaluation per point pair and wavenumber is
// shared by all four operators), accumulating in shared memory in four
// conflict-free phases (a, b), so the result is deterministic.
//
// Quadrature by periodic element distance d: d > near_band tensor Gauss
// (q_far); 2 <= d <= near_band tensor Gauss (q_near); d <= 1 the same q_near
// grid with the log|s - s'| part of each kernel integrated by product
// weights (split K = A log|s - s'| + B, A = -(1/2pi) J0 or -(kappa/2pi) J1 g).
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <complex>
#include <cstring>
#include <vector>

#include "farpair.cuh"
#include "hankel.cuh"
#include "hankeltab.cuh"
#include "internal.h"
#include "split.cuh"

namespace wcs {


template <int OPS>
struct PairSums {
  zd v[OPS][4];  // [operator S~, D, D~, N, D and D~ of the swapped pair][a * 2 + b]
};
using PairOut = PairSums<4>;

__device__ __forceinline__ int periodic_dist(int64_t e, int64_t f, int64_t N) {
  int64_t d = e - f;
  if (d < 0) d = -d;
  if (N - d < d) d = N - d;
  return (int)d;
}

// i/4 * H
__device__ __forceinline__ zd i4(zd H) { return mkz(-0.25 * H.y, 0.25 * H.x); }

// Hankel functions at k R and k~ R
template <bool FROM = false>
__device__ __forceinline__ void hankel_k_kt(const AsmArgs& A, double R, Hankel01& Hk, Hankel01& Ht, int start = 0) {
  if (A.kt_pair) {
    hankel01_pair<FROM>(A.k * R, A.ktp, Hk, Ht, start);
  } else {
    Hk = hankel01(mkz(A.k * R));
    Ht = hankel01(A.kt * R);
  }
}

// FROM (far pairs): the start of the recurrence of each point pair is given (q_far^2 bytes)
template <bool FROM = false>
__device__ void pair_integrals(const AsmArgs& A, int64_t e, int64_t f, PairOut& o, const uint8_t* starts = nullptr) {
#pragma unroll
  for (int op = 0; op < 4; ++op)
#pragma unroll
    for (int j = 0; j < 4; ++j) o.v[op][j] = mkz(0.0);
  const int64_t N = A.N;
  const int d = periodic_dist(e, f, N);
  const double h = A.h, k = A.k, kk2h2 = k * k * h * h;
  const zd kt = A.kt;
  if (d > A.near_band) {
    const int q = A.q_far;
    // Element pairs whose point pairs all lie in the expansion range share
    // the phase and damping of the expansion, evaluated once at the
    // reference argument x0 = k |c_e - c_f| (c: mean of the element's
    // points, every point within 0.45 h of it, so |k R - x0| <= 0.9 k h).
    bool rot = false;
    double x0 = 0.0, damp0 = 0.0;
    zd ph0 = mkz(0.0);
    if (A.kt_pair && A.rot_ok) {
      double cex = 0.0, cey = 0.0, cfx = 0.0, cfy = 0.0;
      for (int p = 0; p < q; ++p) {
        cex += A.far.x[e * q + p];
        cey += A.far.y[e * q + p];
        cfx += A.far.x[f * q + p];
        cfy += A.far.y[f * q + p];
      }
      const double iq = 1.0 / (double)q;
      const double ddx = (cex - cfx) * iq, ddy = (cey - cfy) * iq;
      x0 = k * sqrt(ddx * ddx + ddy * ddy);
      if (x0 >= 20.0 + k * h) {
        rot = true;
        double s0, c0;
        sincos(x0 - 0.25 * WCS_PI, &s0, &c0);
        ph0 = mkz(c0, s0);
        damp0 = exp(-x0 * A.ktp.t);
      }
    }
    for (int p = 0; p < q; ++p) {
      const int64_t ip = e * q + p;
      const double xt = A.far.x[ip], yt = A.far.y[ip], nxt = A.far.nx[ip], nyt = A.far.ny[ip];
      const double xip = A.xf[p], wp = A.wf[p];
      for (int r = 0; r < q; ++r) {
        const int64_t ir = f * q + r;
        const double dx = xt - A.far.x[ir], dy = yt - A.far.y[ir];
        const double nxs = A.far.nx[ir], nys = A.far.ny[ir];
        const double nd = nxt * nxs + nyt * nys;
        Hankel01 Hk, Ht;
        double R, gg;
        if (rot) {
          // one reciprocal square root each for 1/R and for (k R)^-1/2
          const double R2 = dx * dx + dy * dy;
          const double ri = rsqrt(R2);
          R = R2 * ri;
          gg = (dx * nxs + dy * nys) * ri;
          const double x = k * R;
          hankel01_asymptotic_rot(x, rsqrt(x), x0, ph0, damp0, A.ktp, Hk, Ht);
        } else {
          R = sqrt(dx * dx + dy * dy);
          gg = (dx * nxs + dy * nys) / R;
          hankel_k_kt<FROM>(A, R, Hk, Ht, FROM ? starts[p * q + r] : 0);
        }
        const zd gk = i4(Hk.H0);
        const zd gt = i4(Ht.H0);
        const zd dgk = (k * gg) * i4(Hk.H1);
        const zd dgt = gg * (kt * i4(Ht.H1));
        const double w = wp * A.wf[r];
        const double xir = A.xf[r];
        const double ph[2] = {1.0 - xip, xip}, ps[2] = {1.0 - xir, xir};
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
          for (int b = 0; b < 2; ++b) {
            const double c = w * ph[a] * ps[b];
            const double cn = w * ((a == b) ? 1.0 : -1.0) - kk2h2 * nd * c;
            zfmas(o.v[0][a * 2 + b], c, gt);
            zfmas(o.v[1][a * 2 + b], c, dgk);
            zfmas(o.v[2][a * 2 + b], c, dgt);
            zfmas(o.v[3][a * 2 + b], cn, gk);
          }
      }
    }
  } else {
    const int q = A.q_near;
    int kind = -1;
    if (d == 0) kind = 0;
    else if (d == 1) kind = (((e + 1) % N) == f) ? 1 : 2;
    const double* wl = (kind >= 0) ? (A.wlog + kind * q * q) : nullptr;
    const double lh = log(h);
    const zd logkt2 = zlog(0.5 * kt);
    const double logk2 = log(0.5 * k);
    for (int p = 0; p < q; ++p) {
      const int64_t ip = e * q + p;
      const double xt = A.near.x[ip], yt = A.near.y[ip], nxt = A.near.nx[ip], nyt = A.near.ny[ip];
      const double kap = A.near.kappa[ip];
      const double xip = A.xn[p], wp = A.wn[p];
      for (int r = 0; r < q; ++r) {
        const int64_t ir = f * q + r;
        const double xir = A.xn[r];
        const double dx = xt - A.near.x[ir], dy = yt - A.near.y[ir];
        const double nxs = A.near.nx[ir], nys = A.near.ny[ir];
        const double nd = nxt * nxs + nyt * nys;
        const double w = wp * A.wn[r];
        zd kS, kD, kDt, kN;       // smooth parts (full kernels for regular pairs)
        zd aS = mkz(0.0), aD = mkz(0.0), aDt = mkz(0.0), aN = mkz(0.0);  // log coefficients
        double lw = 0.0;          // weight of the log part
        if (kind == 0 && p == r) {
          // coincident points: limits of B = K - A log|s - s'| at R = 0
          kS = mkz(0.0, 0.25) - (1.0 / (2.0 * WCS_PI)) * (logkt2 + mkz(WCS_EULER_GAMMA));
          kN = mkz(-(1.0 / (2.0 * WCS_PI)) * (logk2 + WCS_EULER_GAMMA), 0.25);
          kD = mkz(-kap / (4.0 * WCS_PI));
          kDt = kD;
          aS = mkz(-1.0 / (2.0 * WCS_PI));
          aN = aS;
          lw = wl[p * q + r] + w * lh;
        } else {
          const double R = sqrt(dx * dx + dy * dy);
          const double gg = (dx * nxs + dy * nys) / R;
          Hankel01 Hk, Ht;
          hankel_k_kt(A, R, Hk, Ht);
          kN = i4(Hk.H0);
          kS = i4(Ht.H0);
          kD = (k * gg) * i4(Hk.H1);
          kDt = gg * (kt * i4(Ht.H1));
          if (kind >= 0) {
            double dl = (kind == 0) ? fabs(xip - xir) : ((kind == 1) ? (1.0 - xip + xir) : (xip + 1.0 - xir));
            const double lg = lh + log(dl);  // log |s - s'|
            aS = (-1.0 / (2.0 * WCS_PI)) * Ht.J0;
            aN = (-1.0 / (2.0 * WCS_PI)) * Hk.J0;
            aD = (-(k * gg) / (2.0 * WCS_PI)) * Hk.J1;
            aDt = (-gg / (2.0 * WCS_PI)) * (kt * Ht.J1);
            kS -= lg * aS;
            kN -= lg * aN;
            kD -= lg * aD;
            kDt -= lg * aDt;
            lw = wl[p * q + r] + w * lh;
          }
        }
        const double ph[2] = {1.0 - xip, xip}, ps[2] = {1.0 - xir, xir};
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
          for (int b = 0; b < 2; ++b) {
            const double pp = ph[a] * ps[b];
            const double sab = (a == b) ? 1.0 : -1.0;
            const double c = w * pp;
            const double cn = w * sab - kk2h2 * nd * c;
            zfmas(o.v[0][a * 2 + b], c, kS);
            zfmas(o.v[1][a * 2 + b], c, kD);
            zfmas(o.v[2][a * 2 + b], c, kDt);
            zfmas(o.v[3][a * 2 + b], cn, kN);
            if (kind >= 0) {
              const double cl = lw * pp;
              const double cln = lw * (sab - kk2h2 * nd * pp);
              zfmas(o.v[0][a * 2 + b], cl, aS);
              zfmas(o.v[1][a * 2 + b], cl, aD);
              zfmas(o.v[2][a * 2 + b], cl, aDt);
              zfmas(o.v[3][a * 2 + b], cln, aN);
            }
          }
      }
    }
  }
  const double h2 = h * h;
#pragma unroll
  for (int op = 0; op < 3; ++op)
#pragma unroll
    for (int j = 0; j < 4; ++j) o.v[op][j] = h2 * o.v[op][j];
}


// The operators of a far pair in FP64 from its float-float sums (farpair.cuh).
__device__ __noinline__ void pair_far(const AsmArgs& A, int64_t e, int64_t f, PairSums<6>& out) {
  FarPair<true> o;
  const int q = A.q_far;
  if (q == 4) far_pair<4, true>(A.fc, q, A.fe[e], A.fe[f], A.fp + e * q, A.fp + f * q, o);
  else far_pair<0, true>(A.fc, q, A.fe[e], A.fe[f], A.fp + e * q, A.fp + f * q, o);
  const zd fac[6] = {A.fS, A.fD, A.fDt, A.fN, A.fD, A.fDt};
#pragma unroll
  for (int op = 0; op < 6; ++op)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const ffc v = o.value(op, j);
      out.v[op][j] = fac[op] * mkz((double)v.x.hi + (double)v.x.lo, (double)v.y.hi + (double)v.y.lo);
    }
}

__device__ __forceinline__ bool pair_is_far(const AsmArgs& A, int64_t e, int64_t f) {
  return periodic_dist(e, f, A.N) > A.near_band && far_ok(A.fc, A.fe[e].c, A.fe[f].c);
}

// ----------------------------------------------------------------------------- tables (hankeltab.cuh)
void hankel_tab_args(double t, HankelTabArgs& a) {
  typedef std::complex<double> cd;
  a.t = t;
  const cd c[2] = {cd(1.0, 0.0), cd(1.0, t)};
  for (int w = 0; w < 2; ++w) {
    cd a0 = 1.0, a1 = 0.5 * c[w];   // (-c^2 / 4)^m / m!^2, (c / 2) (-c^2 / 4)^m / (m! (m + 1)!)
    double H = 0.0;
    for (int m = 0; m < HT_M; ++m) {
      if (m > 0) {
        a0 *= -0.25 * c[w] * c[w] / ((double)m * m);
        a1 *= -0.25 * c[w] * c[w] / ((double)m * (m + 1));
        H += 1.0 / m;
      }
      const cd v[4] = {a0, a1, -H * a0, (2.0 * H + 1.0 / (m + 1) - 2.0 * WCS_EULER_GAMMA) * a1};
      for (int j = 0; j < 4; ++j) {
        if (w == 0) a.series[m * 12 + j] = v[j].real();
        else { a.series[m * 12 + 4 + 2 * j] = v[j].real(); a.series[m * 12 + 5 + 2 * j] = v[j].imag(); }
      }
    }
  }
  const cd lc = std::log(c[1]), ic = 1.0 / c[1];
  a.tail[0] = lc.real(); a.tail[1] = lc.imag(); a.tail[2] = ic.real(); a.tail[3] = ic.imag();
  // interpolation at the Chebyshev nodes, as monomials: sum_n (2 - [n = 0]) / D T_n(node_j) T_n(u)
  double T[HT_D][HT_D] = {};   // T[n][power]
  T[0][0] = 1.0;
  T[1][1] = 1.0;
  for (int n = 2; n < HT_D; ++n)
    for (int k = 0; k < HT_D; ++k) T[n][k] = (k > 0 ? 2.0 * T[n - 1][k - 1] : 0.0) - T[n - 2][k];
  for (int j = 0; j < HT_D; ++j) {
    const double th = WCS_PI * (2 * j + 1) / (2.0 * HT_D);
    a.node[j] = std::cos(th);
    for (int k = 0; k < HT_D; ++k) {
      double v = 0.0;
      for (int n = 0; n < HT_D; ++n) v += (n == 0 ? 1.0 : 2.0) / HT_D * std::cos(n * th) * T[n][k];
      a.conv[k * HT_D + j] = v;
    }
  }
}

// J0, J1, Y0, Y1 by the backward recurrence from n = 76 (x < 24), as bessel01_miller_real
__device__ Bessel01 bessel01_long(double x) {
  double jp1 = 0.0, j = 1e-30, norm = 0.0, s0 = 0.0, s1 = 0.0, J1 = 0.0;
  const double iz2 = 2.0 / x;
  for (int n = 76; n > 0; --n) {
    if ((n & 1) == 0) {
      const int k = n >> 1;
      norm += 2.0 * j;
      s0 += ((k & 1) ? -c_recip[k] : c_recip[k]) * j;
    } else {
      const int kp = (n + 1) >> 1, km = (n - 1) >> 1;
      s1 += ((kp & 1) ? -c_recip[kp] : c_recip[kp]) * j;
      if (km >= 1) s1 -= ((km & 1) ? -c_recip[km] : c_recip[km]) * j;
      if (n == 1) J1 = j;
    }
    const double jm = ((double)n * iz2) * j - jp1;
    jp1 = j;
    j = jm;
  }
  const double inv = 1.0 / (norm + j), lz = log(0.5 * x) + WCS_EULER_GAMMA;
  Bessel01 b;
  b.J0 = j * inv;
  b.J1 = J1 * inv;
  b.Y0 = (2.0 / WCS_PI) * (lz * b.J0 - 2.0 * (s0 * inv));
  b.Y1 = (2.0 / WCS_PI) * (lz * b.J1 - b.J0 * (0.5 * iz2) + s1 * inv);
  return b;
}

// one block per interval, the last one copies the series
__global__ void __launch_bounds__(96) k_hankel_table(const __grid_constant__ HankelTabArgs a, double* T) {
  const int b = blockIdx.x, t = threadIdx.x;
  if (b == HT_N) {
    for (int i = t; i < HT_SERIES; i += 96) T[i] = a.series[i];
    if (t < 4) T[HT_SERIES + t] = a.tail[t];
    return;
  }
  __shared__ double v[HT_D][8];
  if (t < HT_D) {
    const double x = HT_X0 + 0.25 + 0.5 * b + 0.25 * a.node[t];
    const Bessel01 f = bessel01_long(x);
    const Hankel01 h = bessel01_shift(x, x * a.t, f);
    v[t][0] = f.J0; v[t][1] = f.Y0; v[t][2] = f.J1; v[t][3] = f.Y1;
    v[t][4] = h.H0.x; v[t][5] = h.H0.y; v[t][6] = h.H1.x; v[t][7] = h.H1.y;
  }
  __syncthreads();
  const int k = t >> 3, fn = t & 7;
  double s = 0.0;
  for (int j = 0; j < HT_D; ++j) s = fma(a.conv[k * HT_D + j], v[j][fn], s);
  T[HT_SERIES + 4 + ((int64_t)b * HT_D + k) * 8 + fn] = s;
}

int64_t hankel_table_doubles() { return HT_SIZE; }

int hankel_table(double t, double* T, cudaStream_t s) {
  HankelTabArgs a;
  hankel_tab_args(t, a);
  k_hankel_table<<<HT_N + 1, 96, 0, s>>>(a, T);
  note_launch();
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) { set_error(std::string("hankel table: ") + cudaGetErrorString(err)); return 3; }
  return 0;
}

// Near-band element pairs (d <= near_band) of the elements e0 .. e0 + ne - 1
// (mod N): the 2 x 2 blocks of the four operators, 32 doubles per pair, pair
// (offset + near_band) * ne + (e - e0).  One warp per pair, the q^2 points over
// its lanes, so that every lane runs the same branch (a thread per pair left 9 of
// 33 lanes of a diagonal tile's warps on the heaviest path in the program, 60 ms
// of FP64 pipe per tile); the 32 sums are joined by a halving exchange that
// leaves sum l in lane l.  Bound: FP64 pipe, ~300 operations a point.
// TAB: Hankel functions from the run's table; without one (k~ off its form, small k a) from
// the full expansions.
template <bool TAB>
__global__ void __launch_bounds__(128) k_near_band(AsmArgs A, int64_t e0, int64_t ne, double* out) {
  const int64_t N = A.N;
  const int64_t pair = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31, nb = A.near_band;
  if (pair >= ne * (2 * nb + 1)) return;
  const int off = (int)(pair / ne) - nb;
  const int64_t e = (e0 + pair % ne) % N, f = ((e + off) % N + N) % N;
  const int q = A.q_near;
  const double h = A.h, k = A.k, kk2h2 = k * k * h * h, lh = log(h);
  const zd kt = A.kt;
  const int d = periodic_dist(e, f, N);
  const int kind = d == 0 ? 0 : (d == 1 ? (((e + 1) % N) == f ? 1 : 2) : -1);
  double v[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = 0.0;
  for (int pt = lane; pt < q * q; pt += 32) {
    const int p = pt / q, r = pt - p * q;
    const int64_t ip = e * q + p, ir = f * q + r;
    const double xip = A.xn[p], xir = A.xn[r], w = A.wn[p] * A.wn[r];
    const double dx = A.near.x[ip] - A.near.x[ir], dy = A.near.y[ip] - A.near.y[ir];
    const double nxs = A.near.nx[ir], nys = A.near.ny[ir];
    const double nd = A.near.nx[ip] * nxs + A.near.ny[ip] * nys;
    zd kS, kD, kDt, kN, aS = mkz(0.0), aD = mkz(0.0), aDt = mkz(0.0), aN = mkz(0.0);
    double lw = 0.0;
    if (kind >= 0) lw = A.wlog[kind * q * q + pt] + w * lh;
    if (kind == 0 && p == r) {
      // coincident points: limits of B = K - A log|s - s'| at R = 0
      const double kap = A.near.kappa[ip];
      kS = mkz(0.0, 0.25) - (1.0 / (2.0 * WCS_PI)) * (zlog(0.5 * kt) + mkz(WCS_EULER_GAMMA));
      kN = mkz(-(1.0 / (2.0 * WCS_PI)) * (log(0.5 * k) + WCS_EULER_GAMMA), 0.25);
      kD = mkz(-kap / (4.0 * WCS_PI));
      kDt = kD;
      aS = mkz(-1.0 / (2.0 * WCS_PI));
      aN = aS;
    } else {
      const double R2 = dx * dx + dy * dy, ri = rsqrt(R2), R = R2 * ri, gg = (dx * nxs + dy * nys) * ri, x = k * R;
      Hankel01 Hk, Ht;
      if (!TAB) {
        hankel_k_kt(A, R, Hk, Ht);
      } else if (x < HT_X0) {
        hankel_tab_series(A.htab, x, log(0.5 * x), Hk, Ht);
      } else if (kind >= 0 || x >= HT_X1) {
        hankel01_pair(x, A.ktp, Hk, Ht);
      } else {
        hankel_tab_poly(A.htab, x, Hk.H0, Hk.H1, Ht.H0, Ht.H1);
      }
      kN = i4(Hk.H0);
      kS = i4(Ht.H0);
      kD = (k * gg) * i4(Hk.H1);
      kDt = gg * (kt * i4(Ht.H1));
      if (kind >= 0) {
        const double dl = (kind == 0) ? fabs(xip - xir) : ((kind == 1) ? (1.0 - xip + xir) : (xip + 1.0 - xir));
        const double lg = lh + log(dl);  // log |s - s'|
        aS = (-1.0 / (2.0 * WCS_PI)) * Ht.J0;
        aN = (-1.0 / (2.0 * WCS_PI)) * Hk.J0;
        aD = (-(k * gg) / (2.0 * WCS_PI)) * Hk.J1;
        aDt = (-gg / (2.0 * WCS_PI)) * (kt * Ht.J1);
        kS -= lg * aS;
        kN -= lg * aN;
        kD -= lg * aD;
        kDt -= lg * aDt;
      }
    }
    const double ph[2] = {1.0 - xip, xip}, ps[2] = {1.0 - xir, xir};
#pragma unroll
    for (int ab = 0; ab < 4; ++ab) {
      const double pp = ph[ab >> 1] * ps[ab & 1], sab = (ab == 0 || ab == 3) ? 1.0 : -1.0;
      const double c = w * pp, cn = w * sab - kk2h2 * nd * c;
      v[2 * ab] = fma(c, kS.x, v[2 * ab]);
      v[2 * ab + 1] = fma(c, kS.y, v[2 * ab + 1]);
      v[8 + 2 * ab] = fma(c, kD.x, v[8 + 2 * ab]);
      v[8 + 2 * ab + 1] = fma(c, kD.y, v[8 + 2 * ab + 1]);
      v[16 + 2 * ab] = fma(c, kDt.x, v[16 + 2 * ab]);
      v[16 + 2 * ab + 1] = fma(c, kDt.y, v[16 + 2 * ab + 1]);
      v[24 + 2 * ab] = fma(cn, kN.x, v[24 + 2 * ab]);
      v[24 + 2 * ab + 1] = fma(cn, kN.y, v[24 + 2 * ab + 1]);
      if (kind >= 0) {   // uniform over the warp
        const double cl = lw * pp, cln = lw * (sab - kk2h2 * nd * pp);
        v[2 * ab] = fma(cl, aS.x, v[2 * ab]);
        v[2 * ab + 1] = fma(cl, aS.y, v[2 * ab + 1]);
        v[8 + 2 * ab] = fma(cl, aD.x, v[8 + 2 * ab]);
        v[8 + 2 * ab + 1] = fma(cl, aD.y, v[8 + 2 * ab + 1]);
        v[16 + 2 * ab] = fma(cl, aDt.x, v[16 + 2 * ab]);
        v[16 + 2 * ab + 1] = fma(cl, aDt.y, v[16 + 2 * ab + 1]);
        v[24 + 2 * ab] = fma(cln, aN.x, v[24 + 2 * ab]);
        v[24 + 2 * ab + 1] = fma(cln, aN.y, v[24 + 2 * ab + 1]);
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const double send = up ? v[i] : v[i + o], keep = up ? v[i + o] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  out[pair * 32 + lane] = lane < 24 ? h * h * v[0] : v[0];
}

int near_band_pairs(const AsmArgs& A, int64_t e0, int64_t ne, double* out, cudaStream_t s) {
  const int64_t pairs = ne * (2 * A.near_band + 1);
  if (A.htab) k_near_band<true><<<(unsigned)((pairs + 3) / 4), 128, 0, s>>>(A, e0, ne, out);
  else k_near_band<false><<<(unsigned)((pairs + 3) / 4), 128, 0, s>>>(A, e0, ne, out);
  note_launch();
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) { set_error(std::string("near band: ") + cudaGetErrorString(err)); return 3; }
  return 0;
}

// The block of a near-band pair from the table of near_band_pairs
__device__ __forceinline__ void pair_near(const double* buf, int64_t e0, int64_t ne, int nb, int64_t N, int64_t e,
                                          int64_t f, PairOut& o) {
  int64_t off = f - e;
  if (off > nb) off -= N;
  else if (off < -nb) off += N;
  const int64_t u = (e - e0 + N) % N;
  const zd* b = (const zd*)(buf + ((off + nb) * ne + u) * 32);
#pragma unroll
  for (int op = 0; op < 4; ++op)
#pragma unroll
    for (int j = 0; j < 4; ++j) o.v[op][j] = b[op * 4 + j];
}

// Element pairs beyond the near band whose point pairs all lie below the table's
// end (T: the table in shared or global memory): the far rule in FP64, the inner
// sums over r shared by both target hats, the kernels' constant factors applied
// to the sums.  OPS = 6 adds D and D~ of the pair (f, e), indexed by (e, f)'s hats:
// the same Hankel values with the other element's normal.
template <int OPS>
__device__ __noinline__ void pair_mid(const AsmArgs& A, const double* T, int64_t e, int64_t f, PairSums<OPS>& o) {
  const int q = A.q_far;
  zd v[OPS][4], vd = mkz(0.0);
#pragma unroll
  for (int i = 0; i < OPS; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) v[i][j] = mkz(0.0);
  for (int p = 0; p < q; ++p) {
    const int64_t ip = e * q + p;
    const double xt = A.far.x[ip], yt = A.far.y[ip], nxt = A.far.nx[ip], nyt = A.far.ny[ip];
    zd u[OPS][2], ud = mkz(0.0);
#pragma unroll
    for (int i = 0; i < OPS; ++i) u[i][0] = u[i][1] = mkz(0.0);
    for (int r = 0; r < q; ++r) {
      const int64_t ir = f * q + r;
      const double dx = xt - A.far.x[ir], dy = yt - A.far.y[ir];
      const double nxs = A.far.nx[ir], nys = A.far.ny[ir];
      const double R2 = dx * dx + dy * dy, ri = rsqrt(R2), x = A.k * (R2 * ri);
      Hankel01 Hk, Ht;
      if (x >= HT_X0) hankel_tab_poly(T, x, Hk.H0, Hk.H1, Ht.H0, Ht.H1);
      else hankel_tab_series(T, x, log(0.5 * x), Hk, Ht);
      const double gg = (dx * nxs + dy * nys) * ri, nd = nxt * nxs + nyt * nys;
      zd K[OPS];
      K[0] = Ht.H0;
      K[1] = gg * Hk.H1;
      K[2] = gg * Ht.H1;
      K[3] = nd * Hk.H0;
      if constexpr (OPS == 6) {
        const double gm = -(dx * nxt + dy * nyt) * ri;
        K[4] = gm * Hk.H1;
        K[5] = gm * Ht.H1;
      }
      const double w1 = A.wf[r] * A.xf[r], w0 = A.wf[r] - w1;
#pragma unroll
      for (int i = 0; i < OPS; ++i) {
        zfmas(u[i][0], w0, K[i]);
        zfmas(u[i][1], w1, K[i]);
      }
      zfmas(ud, A.wf[r], Hk.H0);
    }
    const double w1 = A.wf[p] * A.xf[p], w0 = A.wf[p] - w1;
#pragma unroll
    for (int i = 0; i < OPS; ++i)
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        zfmas(v[i][b], w0, u[i][b]);
        zfmas(v[i][2 + b], w1, u[i][b]);
      }
    zfmas(vd, A.wf[p], ud);
  }
  const double h2 = A.h * A.h, kk2h2 = A.k * A.k * h2;
  const zd fS = mkz(0.0, 0.25 * h2), fD = mkz(0.0, 0.25 * A.k * h2), fDt = mkz(-0.25 * h2 * A.kt.y, 0.25 * h2 * A.kt.x);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    o.v[0][j] = fS * v[0][j];
    o.v[1][j] = fD * v[1][j];
    o.v[2][j] = fDt * v[2][j];
    o.v[3][j] = i4(((j == 0 || j == 3) ? vd : -vd) - kk2h2 * v[3][j]);
    if constexpr (OPS == 6) {
      o.v[4][j] = fD * v[4][j];
      o.v[5][j] = fDt * v[5][j];
    }
  }
}

// True when pair_mid's table covers every point pair of (e, f): centres (of the
// Gauss points) within HT_X1 - 2 k h, points within k h of that (0.9 k h, see pair_integrals).
__device__ __forceinline__ bool pair_is_mid(const AsmArgs& A, int64_t e, int64_t f) {
  const int q = A.q_far;
  const double dx = A.far.x[e * q] - A.far.x[f * q], dy = A.far.y[e * q] - A.far.y[f * q];
  const double lim = HT_X1 - 2.0 * A.k * A.h;
  return lim > 0.0 && A.k * A.k * (dx * dx + dy * dy) < lim * lim;
}

constexpr int TILE = 32;
constexpr int ASM_THREADS = 256;

// One tile of node pairs from FP64 pair integrals: the 33 x 33 element pairs
// that touch it, accumulated in acc[4][TILE][TILE].  pre: the pairs' blocks, already
// integrated.
__device__ __forceinline__ void tile_sums(const AsmArgs& A, int64_t i0, int64_t j0, zd* acc, const zd* pre) {
  const int64_t N = A.N;
  for (int t = threadIdx.x; t < 4 * TILE * TILE; t += blockDim.x) acc[t] = mkz(0.0);
  __syncthreads();
  const int span = TILE + 1;
  const int npairs = span * span;
  for (int base = 0; base < npairs; base += blockDim.x) {
    const int idx = base + threadIdx.x;
    const int el = idx / span, fl = idx - (idx / span) * span;
    bool valid = idx < npairs;
    // element row e = i0 - 1 + el touches node rows i0 - 1 + el + a, a in {0,1}
    // element row i0 - 1 + el feeds tile rows el - 1 (a = 1) and el (a = 0)
    const bool rowok = valid && ((el >= 1 && i0 + el - 1 < N) || (el < TILE && i0 + el < N));
    const bool colok = valid && ((fl >= 1 && j0 + fl - 1 < N) || (fl < TILE && j0 + fl < N));
    PairOut o;
    if (rowok && colok) {
      const int64_t e = ((i0 - 1 + el) % N + N) % N;
      const int64_t f = ((j0 - 1 + fl) % N + N) % N;
      if (A.near_buf && periodic_dist(e, f, N) <= A.near_band) {
        pair_near(A.near_buf, 0, N, A.near_band, N, e, f, o);
      } else if (pre) {
#pragma unroll
        for (int op = 0; op < 4; ++op)
#pragma unroll
          for (int j = 0; j < 4; ++j) o.v[op][j] = pre[(int64_t)idx * 16 + op * 4 + j];
      } else {
        pair_integrals(A, e, f, o);
      }
    }
#pragma unroll
    for (int ph = 0; ph < 4; ++ph) {
      const int a = ph >> 1, b = ph & 1;
      if (rowok && colok) {
        const int li = el - 1 + a, lj = fl - 1 + b;
        if (li >= 0 && li < TILE && lj >= 0 && lj < TILE && i0 + li < N && j0 + lj < N) {
#pragma unroll
          for (int op = 0; op < 4; ++op) acc[(op * TILE + li) * TILE + lj] += o.v[op][ph];
        }
      }
      __syncthreads();
    }
  }
}

// FP64 form.  The tiles around the diagonal hold the near band (144 singular
// points a pair) and the pairs below the expansion range: a CTA of eight warps
// that walks such a tile takes 40 ms while the others take one.  Their pairs are
// integrated by one warp per CTA first (k_assemble_pairs), so that the work spreads
// over the chip; the tile kernel then only sums.  FP64 pipe bound, and a warp pays for
// every branch that one of its lanes takes: near-band rule, recurrence, two expansions.
// So the lanes of a warp hold pairs of one element offset: the near band as a table of
// its own, the tile's far pairs sorted by offset (54 ms at N = 1024 with the pairs in
// tile order, 15 sorted).  The values stay those of the tile order, whose
// recurrences start at the largest index of 32 consecutive pairs: k_pair_starts tables
// these, and in the near band every point below x = 4 starts at 28 in any company
// (band_sorts; otherwise the tile order stays).  The circle's row, a chain of one near-band
// pair's length on a few warps (5.9 ms on its own), runs beside them.
constexpr int PRE_OFF = 3, PRE_SLOTS = 2 * PRE_OFF + 1, PRE_PAIRS = (TILE + 1) * (TILE + 1);

// Slot of tile (ti, tj) in its row's integrated tiles, -1 for the others: tile
// offsets up to PRE_OFF (cyclic) whose element ranges come within 34 elements.
__device__ __forceinline__ int pre_slot(int64_t ti, int64_t tj, int64_t nt, int64_t N) {
  int64_t off = tj - ti;
  if (nt <= PRE_SLOTS) return (int)(off < 0 ? off + nt : off);   // few tiles: all of them
  if (off > PRE_OFF) off -= nt;
  if (off < -PRE_OFF) off += nt;
  if (off < -PRE_OFF || off > PRE_OFF) return -1;
  const int64_t a0 = ti * TILE - 1, a1 = min(N - 1, ti * TILE + TILE - 1), b0 = tj * TILE - 1, b1 = min(N - 1, tj * TILE + TILE - 1);
  const int64_t g1 = ((b0 - a1) % N + N) % N, g2 = ((a0 - b1) % N + N) % N;
  return (off == 0 || min(g1, g2) <= 34) ? (int)(off + PRE_OFF) : -1;
}

// Row 0 of the circle's four operators: node 0 gets element N-1 (a = 1) and element 0
// (a = 0); column j gets elements j-1 (b = 1) and j (b = 0).  One thread per
// (column, element pair); the four partial values are summed in fixed order.
__device__ __forceinline__ void circle_pair(int64_t t, int64_t N, int64_t& e, int64_t& f) {
  const int64_t j = t >> 2;
  e = ((t >> 1) & 1) ? 0 : N - 1;
  f = (t & 1) ? j : (j - 1 + N) % N;
}
__device__ __forceinline__ void circle_store(const PairOut& o, int64_t t, int64_t N, zd* part) {
  const int a = ((t >> 1) & 1) ? 0 : 1, b = (t & 1) ? 0 : 1;
#pragma unroll
  for (int op = 0; op < 4; ++op) {
    const zd v = a ? (b ? o.v[op][3] : o.v[op][2]) : (b ? o.v[op][1] : o.v[op][0]);
    part[(int64_t)op * 4 * N + t] = v;
  }
}

// k R of a near-band point pair is below k h (near_band + 1), its elements' span
__host__ __device__ __forceinline__ bool band_sorts(const AsmArgs& A) {
  return A.kt_pair && A.k * A.h * (A.near_band + 1) < 3.9 && 2 * A.near_band + 1 <= A.N;
}

constexpr unsigned PRE_CHUNKS = (PRE_PAIRS + 31) / 32;

// Column tile of a row's slot, -1 when the slot holds none
__device__ __forceinline__ int64_t pre_tile(int64_t ti, int64_t slot, int64_t nt, int64_t N) {
  int64_t tj = nt <= PRE_SLOTS ? ti + slot : ti + slot - PRE_OFF;
  tj = ((tj % nt) + nt) % nt;
  return slot < nt && pre_slot(ti, tj, nt, N) == slot ? tj : -1;
}

// Element pair (el, fl) of the tile at (i0, j0): false when it touches no node of it
__device__ __forceinline__ bool pre_pair(int64_t i0, int64_t j0, int el, int fl, int64_t N, int64_t& e, int64_t& f) {
  e = ((i0 - 1 + el) % N + N) % N;
  f = ((j0 - 1 + fl) % N + N) % N;
  return ((el >= 1 && i0 + el - 1 < N) || (el < TILE && i0 + el < N)) &&
         ((fl >= 1 && j0 + fl - 1 < N) || (fl < TILE && j0 + fl < N));
}

// First index of the recurrence at every far point pair of 32 consecutive pairs of a tile
__global__ void __launch_bounds__(32) k_pair_starts(const __grid_constant__ AsmArgs A, int64_t nt, int64_t row0,
                                                    uint8_t* starts) {
  const int64_t N = A.N;
  const unsigned id = blockIdx.x, chunk = id % PRE_CHUNKS;
  const int64_t ti = row0 + id / (PRE_CHUNKS * PRE_SLOTS), tj = pre_tile(ti, id / PRE_CHUNKS % PRE_SLOTS, nt, N);
  if (tj < 0) return;
  const int idx = (int)chunk * 32 + threadIdx.x, span = TILE + 1, q = A.q_far;
  int64_t e = 0, f = 0;
  const bool ok = idx < PRE_PAIRS && pre_pair(ti * TILE, tj * TILE, idx / span, idx % span, N, e, f) &&
                  periodic_dist(e, f, N) > A.near_band;
  for (int u = 0; u < q * q; ++u) {
    const int64_t ip = e * q + u / q, ir = f * q + u % q;
    const double dx = A.far.x[ip] - A.far.x[ir], dy = A.far.y[ip] - A.far.y[ir];
    const double x = A.k * sqrt(dx * dx + dy * dy);
    const int n0 = __reduce_max_sync(0xffffffffu, ok && x > 2.0 && x <= 17.0 ? miller_start(x) : 0);
    if (threadIdx.x == 0) starts[(int64_t)id * q * q + u] = (uint8_t)n0;
  }
}

// CTAs: ncirc of the circle B's row (part: 16 N values), nband of the table band, then
// the tiles' far pairs, sorted by offset with the table (starts: k_pair_starts), otherwise
// all pairs in tile order
template <bool SORTED>
__global__ void __launch_bounds__(32) k_assemble_pairs(const __grid_constant__ AsmArgs A, const __grid_constant__ AsmArgs B,
                                                       int64_t nt, int64_t row0, zd* pre, unsigned ncirc, zd* part,
                                                       unsigned nband, zd* band, const uint8_t* starts) {
  const int64_t N = A.N;
  const uint8_t* first = nullptr;
  const int span = TILE + 1;
  unsigned id = blockIdx.x;
  int64_t e = 0, f = 0;
  zd* out = nullptr;               // the pair's block; null: nothing to do
  bool circle = false;
  int64_t t = 0;
  if (id < ncirc) {
    t = (int64_t)id * 32 + threadIdx.x;
    circle = t < 4 * N;
    if (circle) circle_pair(t, N, e, f);
  } else if ((id -= ncirc) < nband) {
    const unsigned nb = (unsigned)((N + 31) / 32);
    const int64_t off = id / nb, u = (int64_t)(id % nb) * 32 + threadIdx.x;
    if (u < N) {
      e = u;
      f = ((e + off - A.near_band) % N + N) % N;
      out = band + (off * N + e) * 16;
    }
  } else {
    id -= nband;
    const int64_t row = id / (PRE_CHUNKS * PRE_SLOTS), ti = row0 + row, slot = id / PRE_CHUNKS % PRE_SLOTS;
    const int64_t tj = pre_tile(ti, slot, nt, N);
    if (tj < 0) return;
    int idx = (int)(id % PRE_CHUNKS) * 32 + threadIdx.x;
    if (idx < PRE_PAIRS) {
      int el = idx / span, fl = idx % span;
      if (SORTED) {   // by fl - el: offsets -32 .. 0 hold 1 .. 33 pairs, their mirror 32 .. 1
        const bool up = idx >= span * (span + 1) / 2;
        const int u = up ? PRE_PAIRS - 1 - idx : idx;
        int d = (int)((sqrtf(8.f * (float)u + 1.f) - 1.f) * 0.5f);
        while (d * (d + 1) / 2 > u) --d;
        while ((d + 1) * (d + 2) / 2 <= u) ++d;
        const int at = u - d * (d + 1) / 2;
        el = up ? at : at + TILE - d;
        fl = up ? at + TILE - d : at;
        idx = el * span + fl;
        first = starts + ((row * PRE_SLOTS + slot) * PRE_CHUNKS + idx / 32) * A.q_far * A.q_far;
      }
      if (pre_pair(ti * TILE, tj * TILE, el, fl, N, e, f) && (!SORTED || periodic_dist(e, f, N) > A.near_band))
        out = pre + (row * PRE_SLOTS + slot) * PRE_PAIRS * 16 + (int64_t)idx * 16;
    }
  }
  if (!circle && !out) return;
  PairOut o;
  if (SORTED && first) pair_integrals<true>(A, e, f, o, first);
  else pair_integrals(circle ? B : A, e, f, o);
  if (circle) {
    circle_store(o, t, N, part);
    return;
  }
#pragma unroll
  for (int op = 0; op < 4; ++op)
#pragma unroll
    for (int j = 0; j < 4; ++j) out[op * 4 + j] = o.v[op][j];
}

// every tile of the rows from row0 on, dense complex output
__global__ void __launch_bounds__(ASM_THREADS) k_assemble(AsmArgs A, int64_t nt, int64_t row0, const zd* pre) {
  extern __shared__ zd acc[];  // [4][TILE][TILE]
  const int64_t N = A.N, ti = row0 + blockIdx.y, tj = blockIdx.x;
  const int64_t i0 = ti * TILE, j0 = tj * TILE;
  const int slot = pre ? pre_slot(ti, tj, nt, N) : -1;
  tile_sums(A, i0, j0, acc,
            slot < 0 ? nullptr : pre + ((int64_t)blockIdx.y * PRE_SLOTS + slot) * PRE_PAIRS * 16);
  zd* outs[4] = {A.S, A.D, A.Dt, A.Nk};
  for (int t = threadIdx.x; t < 4 * TILE * TILE; t += blockDim.x) {
    const int op = t / (TILE * TILE), rem = t - op * TILE * TILE;
    const int li = rem / TILE, lj = rem - (rem / TILE) * TILE;
    if (i0 + li < N && j0 + lj < N) outs[op][(i0 + li) * A.ld + j0 + lj] = acc[t];
  }
}

// Mixed form: the diagonal tiles and the tiles (ti, tj), ti < tj, that k_assemble_far
// listed (those holding an element pair nearer than its route) with their mirror
// images, as split-bf16 planes in both layouts.  S~ and N are symmetric and the Hankel
// values of a pair (e, f) serve (f, e) too, so a listed tile and its mirror are one pass
// (six sums per node pair) and a diagonal tile walks the pairs el <= fl only: that is 5%
// more work a pair on half the pairs (3.1 -> 2.2 ms at N = 2777, 1.5 with the
// pairs in the order of their offset, so that the lanes of a warp take one route).  The sums of a diagonal
// tile's lower half are those of its upper half, as of a tile and its mirror.
// Bound: FP64 pipe.  A listed tile is two jobs of 16 rows, 561 pairs like a diagonal
// tile's, so that a few hundred equal jobs spread evenly over the GPU; 192 threads fill
// 97% of their three rounds, two CTAs a SM, the Hankel table from L1.
constexpr int NEAR_THREADS = 192, NEAR_LD = TILE + 1, NEAR_OPS = 6;
constexpr size_t NEAR_SMEM = sizeof(zd) * NEAR_OPS * TILE * NEAR_LD;

__device__ __forceinline__ void pair_both(const AsmArgs& A, int64_t e, int64_t f, PairSums<6>& o) {
  const int64_t N = A.N;
  const bool band = A.near_buf && periodic_dist(e, f, N) <= A.near_band;
  if (!band && pair_is_far(A, e, f)) { pair_far(A, e, f, o); return; }
  if (!band && A.htab && pair_is_mid(A, e, f)) { pair_mid<6>(A, A.htab, e, f, o); return; }
  PairOut p;
  for (int m = 0; m < 2; ++m) {
    const int64_t x = m ? f : e, y = m ? e : f;
    if (band) pair_near(A.near_buf, 0, N, A.near_band, N, x, y, p);
    else pair_integrals(A, x, y, p);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (m) {
        o.v[4][j] = p.v[1][(j & 1) * 2 + (j >> 1)];
        o.v[5][j] = p.v[2][(j & 1) * 2 + (j >> 1)];
      } else {
#pragma unroll
        for (int op = 0; op < 4; ++op) o.v[op][j] = p.v[op][j];
      }
    }
  }
}

__global__ void __launch_bounds__(NEAR_THREADS, 2) k_assemble_near(AsmArgs A, int64_t nt) {
  extern __shared__ zd acc[];  // [6][TILE][NEAR_LD], later the packed planes
  const int64_t N = A.N;
  const int64_t jobs = nt + 2 * ((int64_t)A.tile_list[0] - nt);
  const int span = TILE + 1;
  // the pairs of a half tile in the order of their offset fl - el = k - TILE / 2, so that
  // the lanes of a warp take one route (tabulated, far or near band)
  __shared__ uint16_t order[(TILE / 2 + 1) * (TILE + 1)];
  for (int t = threadIdx.x; t < (TILE / 2 + 1) * span; t += NEAR_THREADS) {
    constexpr int H = TILE / 2;              // diagonals of 1 .. H + 1, H times H + 1, H + 1 .. 1 pairs
    const int el = t / span, fl = t - el * span, k = fl - el + H;
    const int before = k <= H ? k * (k + 1) / 2
                              : (k <= TILE ? H * (H + 1) / 2 + (H + 1) * (k - H)
                                           : (H + 1) * (TILE + 1) - (TILE + H + 1 - k) * (TILE + H + 2 - k) / 2);
    order[before + min(el, fl)] = (uint16_t)t;
  }
  for (int64_t u = blockIdx.x; u < jobs; u += gridDim.x) {
    const bool diag = u < nt;
    const int64_t tile = diag ? u * nt + u : A.tile_list[1 + nt + ((u - nt) >> 1)];
    const int rows = diag ? TILE : TILE / 2;
    const int64_t i0 = (tile / nt) * TILE + (diag ? 0 : ((u - nt) & 1) * rows), j0 = (tile % nt) * TILE;
    if (i0 >= N) continue;
    const int npairs = diag ? span * (span + 1) / 2 : (rows + 1) * span;
    for (int t = threadIdx.x; t < NEAR_OPS * TILE * NEAR_LD; t += NEAR_THREADS) acc[t] = mkz(0.0);
    __syncthreads();
    for (int base = 0; base < npairs; base += NEAR_THREADS) {
      const int idx = base + threadIdx.x;
      int el, fl;
      if (diag) {   // offsets fl - el = 32 .. 0 hold 1 .. 33 pairs
        int d = (int)((sqrtf(8.f * (float)idx + 1.f) - 1.f) * 0.5f);
        while (d * (d + 1) / 2 > idx) --d;
        while ((d + 1) * (d + 2) / 2 <= idx) ++d;
        el = idx - d * (d + 1) / 2;
        fl = el + TILE - d;
      } else {
        const int t = idx < npairs ? order[idx] : 0;
        el = t / span;
        fl = t - el * span;
      }
      // element row e = i0 - 1 + el feeds tile rows el - 1 (a = 1) and el (a = 0)
      const bool valid = idx < npairs;
      const bool rowok = valid && ((el >= 1 && i0 + el - 1 < N) || (el < rows && i0 + el < N));
      const bool colok = valid && ((fl >= 1 && j0 + fl - 1 < N) || (fl < TILE && j0 + fl < N));
      PairSums<6> o;
      if (rowok && colok) {
        const int64_t e = ((i0 - 1 + el) % N + N) % N;
        const int64_t f = ((j0 - 1 + fl) % N + N) % N;
        pair_both(A, e, f, o);
      }
#pragma unroll
      for (int ph = 0; ph < 4; ++ph) {
        const int a = ph >> 1, b = ph & 1;
        const int li = el - 1 + a, lj = fl - 1 + b;
        // a diagonal tile's sums live on and above its diagonal: a pair el < fl adds its
        // swapped pair's share on the diagonal, a pair el = fl leaves out its lower corner
        const bool ok = rowok && colok && li >= 0 && li < rows && lj >= 0 && lj < TILE && i0 + li < N && j0 + lj < N &&
                        !(diag && li > lj);
        if (ok) {
          zd* c = acc + li * NEAR_LD + lj;
          const bool twice = diag && li == lj && el < fl;
#pragma unroll
          for (int op = 0; op < 4; ++op) {
            zd v = o.v[op][ph];
            if (twice) v += (op == 1 || op == 2) ? o.v[op + 3][ph] : v;
            c[op * TILE * NEAR_LD] += v;
          }
#pragma unroll
          for (int op = 4; op < 6; ++op) c[op * TILE * NEAR_LD] += o.v[op][ph];
        }
        __syncthreads();
      }
    }
    // entries as packed planes, in place
    for (int t = threadIdx.x; t < NEAR_OPS * rows * TILE; t += NEAR_THREADS) {
      zd* slot = acc + (t / (rows * TILE) * TILE + t / TILE % rows) * NEAR_LD + t % TILE;
      const zd v = *slot;
      uint16_t re[3] = {0, 0, 0}, im[3] = {0, 0, 0};
      split3_bits(v.x, A.planes, &re[0], &re[1], &re[2]);
      split3_bits(v.y, A.planes, &im[0], &im[1], &im[2]);
      uint4 w;
      w.x = (uint32_t)re[0] | ((uint32_t)im[0] << 16);
      w.y = (uint32_t)re[1] | ((uint32_t)im[1] << 16);
      w.z = (uint32_t)re[2] | ((uint32_t)im[2] << 16);
      w.w = 0u;
      *(uint4*)slot = w;
    }
    __syncthreads();
    // layout 0: row i holds (re, im) of column j at 2 j; layout 1 (transpose): row j
    // holds entry (i, j) at 2 i; consecutive threads walk the contiguous index.  Entry
    // (j, i) of operator x comes from x (S~, N) or from the swapped pair's sums.
    auto at = [&](int op, int li, int lj) {
      return *(const uint4*)(acc + ((size_t)op * TILE + li) * NEAR_LD + lj);
    };
    auto put = [&](int op, int lay, int64_t off, const uint4& w) {
      const uint32_t p[3] = {w.x, w.y, w.z};
#pragma unroll
      for (int q = 0; q < 3; ++q)
        if (q < A.planes) *(uint32_t*)(A.P[op][lay][q] + off) = p[q];
    };
    for (int t = threadIdx.x; t < 4 * rows * TILE; t += NEAR_THREADS) {
      const int op = t / (rows * TILE), rem = t - op * rows * TILE;
      const int mop = (op == 1 || op == 2) ? op + 3 : op;
      if (diag) {
        const int x = rem / TILE, y = rem % TILE;
        if (i0 + x < N && j0 + y < N) {
          const int64_t off = (i0 + x) * A.ldp + 2 * (j0 + y);
          put(op, 0, off, x <= y ? at(op, x, y) : at(mop, y, x));    // entry (x, y)
          put(op, 1, off, y <= x ? at(op, y, x) : at(mop, x, y));    // entry (y, x)
        }
      } else {
        int li = rem / TILE, lj = rem % TILE;   // along j for fixed i
        if (i0 + li < N && j0 + lj < N) {
          const int64_t off = (i0 + li) * A.ldp + 2 * (j0 + lj);
          put(op, 0, off, at(op, li, lj));
          put(op, 1, off, at(mop, li, lj));
        }
        lj = rem / rows;                        // along i for fixed j
        li = rem % rows;
        if (i0 + li < N && j0 + lj < N) {
          const int64_t off = (j0 + lj) * A.ldp + 2 * (i0 + li);
          put(op, 1, off, at(op, li, lj));
          put(op, 0, off, at(mop, li, lj));
        }
      }
    }
    __syncthreads();
  }
}

__global__ void k_circle_row_part(AsmArgs A, zd* part) {
  const int64_t N = A.N;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 4 * N) return;
  int64_t e, f;
  circle_pair(t, N, e, f);
  PairOut o;
  if (A.near_buf && periodic_dist(e, f, N) <= A.near_band) pair_near(A.near_buf, N - 1, 2, A.near_band, N, e, f, o);
  else if (A.htab && pair_is_mid(A, e, f)) pair_mid<4>(A, A.htab, e, f, o);
  else pair_integrals(A, e, f, o);
  circle_store(o, t, N, part);
}

__global__ void k_circle_row_sum(AsmArgs A, const zd* part) {
  const int64_t N = A.N;
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= N) return;
  zd* outs[4] = {A.S, A.D, A.Dt, A.Nk};
  for (int op = 0; op < 4; ++op) {
    const zd* p = part + (int64_t)op * 4 * N + 4 * j;
    outs[op][j] = ((p[0] + p[1]) + p[2]) + p[3];
  }
}

// Entries (row i, col j): sum of the four element pairs (i-1|i) x (j-1|j).
__global__ void k_entries(AsmArgs A, int64_t count, const int64_t* rows, const int64_t* cols,
                          zd* out4) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= count) return;
  const int64_t N = A.N, i = rows[t], j = cols[t];
  zd sum[4] = {mkz(0.0), mkz(0.0), mkz(0.0), mkz(0.0)};
  for (int a = 0; a < 2; ++a)
    for (int b = 0; b < 2; ++b) {
      const int64_t e = (i - a + N) % N, f = (j - b + N) % N;
      PairOut o;
      pair_integrals(A, e, f, o);
      for (int op = 0; op < 4; ++op) sum[op] += o.v[op][a * 2 + b];
    }
  for (int op = 0; op < 4; ++op) out4[op * count + t] = sum[op];
}

// Coefficient tables of hankel01_asymptotic_fixed for k~ = k (1 + i t), and
// the x above which 2M terms (M = 2, 3, 4, 5, 7) meet the relative tolerance
// tol: the first omitted term max_nu |a_2M(nu)| / x^2M (|1 + i t|^-2M <= 1),
// with 10% margin on x and never below 20, where the expansion starts
void fill_asymptotic(KtPair& kp, double tol) {
  AsymCoef& h = kp.asym;
  std::memset(&h, 0, sizeof(h));
  const std::complex<double> c1 = std::complex<double>(1.0, 0.0) / std::complex<double>(1.0, kp.t);
  for (int nu = 0; nu < 2; ++nu) {
    double a = 1.0;
    std::complex<double> cp = 1.0;   // c1^k
    for (int k = 0; k < 2 * ASYM_M; ++k) {
      if (k > 0) {
        a *= (4.0 * nu * nu - (2.0 * k - 1.0) * (2.0 * k - 1.0)) / (8.0 * k);
        cp *= c1;
      }
      const int m = k / 2;
      const double sg = (m & 1) ? -1.0 : 1.0;
      const std::complex<double> b = sg * a * cp;
      if ((k & 1) == 0) { h.re[nu][m] = sg * a; h.ce[nu][m] = mkz(b.real(), b.imag()); }
      else { h.ro[nu][m] = sg * a; h.co[nu][m] = mkz(b.real(), b.imag()); }
    }
  }
  const int Ms[5] = {2, 3, 4, 5, 7};
  for (int i = 0; i < 5; ++i) {
    const int k2 = 2 * Ms[i];
    double need = 20.0;
    for (int nu = 0; nu < 2; ++nu) {
      double a = 1.0;
      for (int k = 1; k <= k2; ++k) a *= (4.0 * nu * nu - (2.0 * k - 1.0) * (2.0 * k - 1.0)) / (8.0 * k);
      need = std::max(need, 1.1 * std::pow(std::fabs(a) / tol, 1.0 / k2));
    }
    kp.xth[i] = need;
  }
}

static size_t pre_bytes(int64_t N) {
  const int64_t rows = std::min<int64_t>((N + TILE - 1) / TILE, 128);
  return sizeof(zd) * 16 * PRE_PAIRS * PRE_SLOTS * (size_t)rows;
}

static size_t band_bytes(const AsmArgs& A) {
  const size_t band = sizeof(zd) * 16 * (size_t)A.N * (size_t)(2 * A.near_band + 1);
  return band_sorts(A) && band <= ((size_t)1 << 30) ? band : 0;
}

size_t assemble_dense_bytes(const AsmArgs& A) {
  const int64_t rows = std::min<int64_t>((A.N + TILE - 1) / TILE, 128);
  const size_t starts = (size_t)rows * PRE_SLOTS * PRE_CHUNKS * A.q_far * A.q_far;
  return pre_bytes(A.N) + (band_bytes(A) > 0 ? band_bytes(A) + starts : 0);
}

int assemble_dense(AsmArgs A, const AsmArgs& B, zd* part, void* ws, cudaStream_t s) {
  const size_t smem = sizeof(zd) * 4 * TILE * TILE;
  cudaFuncSetAttribute(k_assemble, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  const int64_t nt = (A.N + TILE - 1) / TILE;
  zd* pre = (zd*)ws;
  unsigned ncirc = 0, nband = 0;
  uint8_t* starts = nullptr;
  if (ws) {
    ncirc = (unsigned)((4 * A.N + 31) / 32);
    if (band_bytes(A) > 0) {
      A.near_buf = (const double*)((char*)ws + pre_bytes(A.N));
      starts = (uint8_t*)A.near_buf + band_bytes(A);
      nband = (unsigned)((A.N + 31) / 32 * (2 * A.near_band + 1));
    }
  } else {
    k_circle_row_part<<<(unsigned)((4 * A.N + 63) / 64), 64, 0, s>>>(B, part);
    note_launch();
  }
  // 128 rows of tiles at a time bound the blocks kept (250 MB)
  for (int64_t r0 = 0; r0 < nt; r0 += 128) {
    const unsigned rows = (unsigned)std::min<int64_t>(128, nt - r0), far = PRE_CHUNKS * PRE_SLOTS * rows;
    if (ws) {
      if (r0 > 0) ncirc = nband = 0;
      if (starts) {
        k_pair_starts<<<far, 32, 0, s>>>(A, nt, r0, starts);
        note_launch();
        k_assemble_pairs<true><<<ncirc + nband + far, 32, 0, s>>>(A, B, nt, r0, pre, ncirc, part, nband, (zd*)A.near_buf, starts);
      } else {
        k_assemble_pairs<false><<<ncirc + far, 32, 0, s>>>(A, B, nt, r0, pre, ncirc, part, 0, nullptr, nullptr);
      }
      note_launch();
    }
    k_assemble<<<dim3((unsigned)nt, rows), ASM_THREADS, smem, s>>>(A, nt, r0, pre);
    note_launch();
  }
  k_circle_row_sum<<<(unsigned)((A.N + 127) / 128), 128, 0, s>>>(B, part);
  note_launch();
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) { set_error(std::string("assemble: ") + cudaGetErrorString(err)); return 3; }
  return 0;
}

// float-float helpers for the epilogue of k_assemble_far
struct ff2 {
  ff r, i;
};
__device__ __forceinline__ ff2 ff2_of(zd z) { return ff2{ff_of(z.x), ff_of(z.y)}; }
// bf16 planes of a float-float value: hi - bf16(hi) is exact in FP32, so the
// second residual carries the value to ~2^-24 of the first plane's scale
__device__ __forceinline__ void ff_planes(ff x, uint16_t (&p)[3]) {
  const __nv_bfloat16 h0 = __float2bfloat16_rn(x.hi);
  const float r1 = (x.hi - __bfloat162float(h0)) + x.lo;
  const __nv_bfloat16 h1 = __float2bfloat16_rn(r1);
  const float r2 = r1 - __bfloat162float(h1);
  p[0] = __bfloat16_as_ushort(h0);
  p[1] = __bfloat16_as_ushort(h1);
  p[2] = __bfloat16_as_ushort(__float2bfloat16_rn(r2));
}
// Tiles whose element pairs all take the FP32 route of farpair.cuh; a tile with
// a nearer pair is put on the list of k_assemble_near instead.  A CTA owns the
// tile (ti, tj), ti < tj, and its mirror image (the diagonal tiles are never
// far): S~ and N are symmetric and every Hankel evaluation serves both.  One
// thread per element pair, the pair's values added into float-float sums per
// node pair in shared memory in four conflict-free phases, then multiplied by
// their FP64 factors (as float-float), split into bf16 planes once and written in
// both layouts of both tiles.
// Bound: FP32 issue.  384 threads: three warps per scheduler at 168 registers,
// and 1089 pairs fill 95% of three rounds (256 threads: 85% of five).
constexpr int FAR_THREADS = 384, FAR_LD = TILE + 1, FAR_OPS = 6;
constexpr size_t FAR_SMEM = sizeof(float4) * FAR_OPS * TILE * FAR_LD;

template <int Q>
__global__ void __launch_bounds__(FAR_THREADS, 1) k_assemble_far(AsmArgs A, int64_t nt) {
  extern __shared__ float4 facc[];   // [6][TILE][FAR_LD] (re hi, re lo, im hi, im lo), later the planes
  // blockIdx.x -> (ti, tj), ti < tj: row tj of the lower triangle holds tj tiles
  const int64_t u0 = blockIdx.x;
  int64_t tj = (int64_t)((1.0 + sqrt(1.0 + 8.0 * (double)u0)) * 0.5);
  while (tj * (tj - 1) / 2 > u0) --tj;
  while ((tj + 1) * tj / 2 <= u0) ++tj;
  const int64_t ti = u0 - tj * (tj - 1) / 2;
  const int64_t N = A.N;
  const int64_t i0 = ti * TILE, j0 = tj * TILE;
  const int span = TILE + 1;
  const int npairs = span * span;
  int near = 0;
  for (int u = threadIdx.x; u < npairs; u += FAR_THREADS) {
    const int el = u / span, fl = u - (u / span) * span;
    int64_t e = i0 - 1 + el, f = j0 - 1 + fl;
    if (e < 0) e += N;
    if (e >= N) e -= N;
    if (f >= N) f -= N;
    if (!pair_is_far(A, e, f)) near = 1;
  }
  for (int t = threadIdx.x; t < FAR_OPS * TILE * FAR_LD; t += FAR_THREADS) facc[t] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (__syncthreads_or(near)) {
    if (threadIdx.x == 0) {
      A.tile_list[1 + atomicAdd(A.tile_list, 1)] = (int)(ti * nt + tj);
    }
    return;
  }
  for (int base = 0; base < npairs; base += FAR_THREADS) {
    const int idx = base + threadIdx.x;
    const int el = idx / span, fl = idx - (idx / span) * span;
    const bool valid = idx < npairs;
    const bool rowok = valid && ((el >= 1 && i0 + el - 1 < N) || (el < TILE && i0 + el < N));
    const bool colok = valid && ((fl >= 1 && j0 + fl - 1 < N) || (fl < TILE && j0 + fl < N));
    FarPair<true> o;
    if (rowok && colok) {
      int64_t e = i0 - 1 + el, f = j0 - 1 + fl;
      if (e < 0) e += N;
      const int q = Q ? Q : A.q_far;
      far_pair<Q, true>(A.fc, q, A.fe[e], A.fe[f], A.fp + e * q, A.fp + f * q, o);
    }
#pragma unroll
    for (int ph = 0; ph < 4; ++ph) {
      const int a = ph >> 1, b = ph & 1;
      if (rowok && colok) {
        const int li = el - 1 + a, lj = fl - 1 + b;
        if (li >= 0 && li < TILE && lj >= 0 && lj < TILE && i0 + li < N && j0 + lj < N) {
#pragma unroll
          for (int op = 0; op < FAR_OPS; ++op) {
            const ffc v = o.value(op, ph);
            float4 s = facc[(op * TILE + li) * FAR_LD + lj];
            const ff x = ff_two_sum(s.x, v.x.hi), y = ff_two_sum(s.z, v.y.hi);
            s.x = x.hi;
            s.y += x.lo + v.x.lo;
            s.z = y.hi;
            s.w += y.lo + v.y.lo;
            facc[(op * TILE + li) * FAR_LD + lj] = s;
          }
        }
      }
      __syncthreads();
    }
  }
  // entries: the FP64 run factors times the tile sums, in float-float on the
  // FP32 pipe (~44 bits; the FP64 pipe is 64 times slower), as packed planes
  const ff2 fac[4] = {ff2_of(A.fS), ff2_of(A.fD), ff2_of(A.fDt), ff2_of(A.fN)};
#pragma unroll
  for (int op = 0; op < FAR_OPS; ++op) {
    const ff2 fo = fac[op < 4 ? op : op - 3];
    for (int u = threadIdx.x; u < TILE * TILE; u += FAR_THREADS) {
      float4& slot = facc[(op * TILE + u / TILE) * FAR_LD + u % TILE];
      const float4 s = slot;
      const ff ar = ff_quick(s.x, s.y), ai = ff_quick(s.z, s.w);
      uint16_t re[3], im[3];
      ff_planes(ff_add(ff_mul(fo.r, ar), ff_neg(ff_mul(fo.i, ai))), re);
      ff_planes(ff_add(ff_mul(fo.r, ai), ff_mul(fo.i, ar)), im);
      uint4 w;
      w.x = (uint32_t)re[0] | ((uint32_t)im[0] << 16);
      w.y = (uint32_t)re[1] | ((uint32_t)im[1] << 16);
      w.z = (uint32_t)re[2] | ((uint32_t)im[2] << 16);
      w.w = 0u;
      *(uint4*)&slot = w;
    }
  }
  __syncthreads();
  // stored operator x: entry (i, j) from accumulator x; entry (j, i) from x (S~,
  // N) or from the mirrored accumulator.  "wide" rows run along j for fixed i
  // (layout 0 of (i, j), layout 1 of (j, i)), "tall" ones along i for fixed j.
  for (int u = threadIdx.x; u < 4 * TILE * TILE; u += FAR_THREADS) {
    const int op = u / (TILE * TILE), rem = u - op * TILE * TILE;
    const int x = rem / TILE, y = rem - (rem / TILE) * TILE;
    const int mop = (op == 1 || op == 2) ? op + 3 : op;
    if (i0 + x < N && j0 + y < N) {     // wide: li = x, lj = y
      const int64_t off = (i0 + x) * A.ldp + 2 * (j0 + y);
      const uint4 d = *(const uint4*)&facc[(op * TILE + x) * FAR_LD + y];
      const uint4 m = *(const uint4*)&facc[(mop * TILE + x) * FAR_LD + y];
      const uint32_t dv[3] = {d.x, d.y, d.z}, mv[3] = {m.x, m.y, m.z};
#pragma unroll
      for (int q = 0; q < 3; ++q)
        if (q < A.planes) {
          *(uint32_t*)(A.P[op][0][q] + off) = dv[q];
          *(uint32_t*)(A.P[op][1][q] + off) = mv[q];
        }
    }
    if (i0 + y < N && j0 + x < N) {     // tall: li = y, lj = x
      const int64_t off = (j0 + x) * A.ldp + 2 * (i0 + y);
      const uint4 d = *(const uint4*)&facc[(op * TILE + y) * FAR_LD + x];
      const uint4 m = *(const uint4*)&facc[(mop * TILE + y) * FAR_LD + x];
      const uint32_t dv[3] = {d.x, d.y, d.z}, mv[3] = {m.x, m.y, m.z};
#pragma unroll
      for (int q = 0; q < 3; ++q)
        if (q < A.planes) {
          *(uint32_t*)(A.P[op][1][q] + off) = dv[q];
          *(uint32_t*)(A.P[op][0][q] + off) = mv[q];
        }
    }
  }
}

// the diagonal tiles open the list of the FP64 kernel
__global__ void k_diag_tiles(int* list, int64_t nt) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t == 0) list[0] = (int)nt;
  if (t < nt) list[1 + t] = (int)(t * nt + t);
}

int assemble_planes(const AsmArgs& A, cudaStream_t s, cudaEvent_t* mid, int64_t* fp64_tiles, int64_t* tiles) {
  cudaFuncSetAttribute(k_assemble_near, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)NEAR_SMEM);
  cudaFuncSetAttribute(k_assemble_far<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FAR_SMEM);
  cudaFuncSetAttribute(k_assemble_far<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FAR_SMEM);
  const int64_t nt = (A.N + TILE - 1) / TILE;
  k_diag_tiles<<<(unsigned)((nt + 127) / 128), 128, 0, s>>>(A.tile_list, nt);
  note_launch();
  if (nt > 1) {
    const unsigned grid = (unsigned)(nt * (nt - 1) / 2);
    if (A.q_far == 4) k_assemble_far<4><<<grid, FAR_THREADS, FAR_SMEM, s>>>(A, nt);
    else k_assemble_far<0><<<grid, FAR_THREADS, FAR_SMEM, s>>>(A, nt);
    note_launch();
  }
  if (mid) { cudaEventRecord(mid[0], s); cudaEventRecord(mid[1], s); }
  k_assemble_near<<<(unsigned)std::min<int64_t>(nt * nt, 152 * 2), NEAR_THREADS, NEAR_SMEM, s>>>(A, nt);
  note_launch();
  if (fp64_tiles) {   // the tiles that took the FP64 kernel (for the work count of each kernel)
    int n = 0;
    cudaMemcpyAsync(&n, A.tile_list, sizeof(int), cudaMemcpyDeviceToHost, s);
    cudaStreamSynchronize(s);
    *fp64_tiles = 2 * (int64_t)n - nt;   // the list holds one of a tile and its mirror
    *tiles = nt * nt;
  }
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) { set_error(std::string("assemble (planes): ") + cudaGetErrorString(err)); return 3; }
  return 0;
}

__global__ void k_far_tables(AsmArgs A, Points cen, FarElem* fe, FarPoint* fp) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int q = A.q_far;
  const Points& far = A.far;
  const double h = A.h;
  if (t >= A.N * q) return;
  const int64_t e = t / q;
  const int p = (int)(t - e * q);
  fp[t] = far_point(cen.x[e], cen.y[e], cen.nx[e], cen.ny[e], far.x[t], far.y[t], far.nx[t], far.ny[t], h,
                    A.xf[p] - 0.5);
  if (p == 0) fe[e] = far_elem(cen.x[e], cen.y[e], cen.nx[e], cen.ny[e]);
}

int far_tables(const AsmArgs& A, const Points& cen, FarElem* fe, FarPoint* fp, cudaStream_t s) {
  const int64_t n = A.N * A.q_far;
  k_far_tables<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(A, cen, fe, fp);
  note_launch();
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) { set_error(std::string("far tables: ") + cudaGetErrorString(err)); return 3; }
  return 0;
}

int assemble_circle_row(const AsmArgs& A, zd* part, cudaStream_t s) {
  k_circle_row_part<<<(unsigned)((4 * A.N + 63) / 64), 64, 0, s>>>(A, part);
  note_launch();
  k_circle_row_sum<<<(unsigned)((A.N + 127) / 128), 128, 0, s>>>(A, part);
  note_launch();
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) { set_error(std::string("circle row: ") + cudaGetErrorString(err)); return 3; }
  return 0;
}

int assemble_entries(const AsmArgs& A, int64_t count, const int64_t* rows, const int64_t* cols,
                     zd* out4, cudaStream_t s) {
  if (count <= 0) return 0;
  k_entries<<<(unsigned)((count + 63) / 64), 64, 0, s>>>(A, count, rows, cols, out4);
  note_launch();
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) { set_error(std::string("entries: ") + cudaGetErrorString(err)); return 3; }
  return 0;
}


// ---------------------------------------------------------------------------
// Shape derivatives of the Galerkin entries (differentiation of Sec. II Eq. 4
// with respect to the contour).  A far entry is h^2 sum w_p w_r phi_a phi_b K
// over point pairs; moving the contour moves the points (r, r'), turns the
// normals (n, n'), changes k~ through a = L / 2 pi (Sec. III) and scales h^2.
// For the forms T = sum_ij W_ij X_ij the derivative with respect to any
// parameter is therefore
//   sum_P (dT/dr_P . dr_P/dp + dT/dn_P . dn_P/dp) + dT/dk~ dk~/dp + 2 (dh/h) T_h2,
// and one pass over the point pairs gathers dT/dr_P, dT/dn_P (per point),
// dT/dk~ and T_h2 for all parameters at once.  Kernel derivatives, with
// d = r - r', R = |d|, d^ = d / R, g = d.n' / R, z = kappa R,
// H1'(z) = H0(z) - H1(z) / z:
//   S~ = (i/4) H0(k~R):      d/dd = -(i/4) k~ H1 d^,   d/dk~ = -(i/4) R H1
//   D  = (i k/4) H1(kR) g:   d/dd = (i k/4) [k H1' g d^ + H1 (n' - g d^) / R],
//                            d/dn' = (i k/4) H1 d^
//   D~ likewise with k~, and d/dk~ = (i/4) k~ R H0(k~R) g
//   N  (Maue form): [s_a s_b - k^2 h^2 (n.n') phi_a phi_b] (i/4) H0(kR):
//                            d/dd = -(i/4) k H1 d^ (both parts),
//                            d/dn = (i/4) H0 n' and d/dn' = (i/4) H0 n (second part)
// Only far pairs are differentiated here; the near band keeps its singular
// product rules and is differenced (shape_near_forms).
// ---------------------------------------------------------------------------
constexpr int SH_E = 2;       // element rows per block
constexpr int SH_W = 4;       // warps per block, 32 element columns each

// Bound: FP64 pipe.  The pair's coefficients are folded into the Hankel values first
// (k into D's, k~ into D~'s, so H1' = H0 - H1 / z needs no division), the common factor
// i/4 is applied to the sums, and the eight row sums of a point pair cross the warp by a
// halving exchange (9 additions instead of 40) into the warp's own accumulators:
// 111 -> 76 ms at N = 1024, q = 6, and 47 with blocks of two rows, the longest first.
__global__ void __launch_bounds__(32 * SH_W) k_shape_far(ShapeArgs S) {
  const AsmArgs& A = S.A;
  const int64_t N = A.N;
  const int q = A.q_far;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // the column blocks in the order of their distance from the diagonal, whose pairs (the
  // recurrences below x = 17) take several times longer than the others, 27 ms a warp at
  // eight rows: short blocks, the long ones first
  const int64_t e0 = (int64_t)blockIdx.x * SH_E, nf = gridDim.y;
  const int64_t off = (blockIdx.y & 1) ? (int64_t)(blockIdx.y + 1) / 2 : nf - (int64_t)blockIdx.y / 2;
  const int64_t f = (e0 / (32 * SH_W) + off) % nf * (32 * SH_W) + threadIdx.x;
  const bool fvalid = f < N;
  __shared__ double rowacc[SH_W][SH_E][16][8];
  __shared__ double red[SH_W][4];
  for (int t = threadIdx.x; t < SH_W * SH_E * 16 * 8; t += 32 * SH_W) (&rowacc[0][0][0][0])[t] = 0.0;
  __syncthreads();
  const double h = A.h, k = A.k, h2 = h * h, kk2h2 = k * k * h2;
  const zd kt = A.kt;
  const int own = ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);   // row sum left in the lane
  double sc[4] = {0.0, 0.0, 0.0, 0.0};
  const int64_t f1 = fvalid ? (f + 1) % N : 0;
  for (int r = 0; r < q; ++r) {
    double col[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    const int64_t iq = fvalid ? f * q + r : 0;
    const double xq = A.far.x[iq], yq = A.far.y[iq], nxq = A.far.nx[iq], nyq = A.far.ny[iq];
    const double eta = A.xf[r], wr = A.wf[r];
    const double pb0 = 1.0 - eta, pb1 = eta;
    for (int el = 0; el < SH_E; ++el) {
      const int64_t e = e0 + el;
      const bool ok = fvalid && e < N && periodic_dist(e, f, N) > A.near_band;
      if (!__any_sync(0xffffffffu, ok)) continue;
      // per operator: sum_b W(e + a, f + b) phi_b(eta_r) for a = 0, 1, times its share of
      // the point pair's factor; for the derivative part of N, sum_ab s_a s_b W_N(e + a, f + b)
      zd cw[4][2], cd = mkz(0.0);
#pragma unroll
      for (int X = 0; X < 4; ++X) cw[X][0] = cw[X][1] = mkz(0.0);
      if (ok) {
        const int64_t ea[2] = {e, (e + 1) % N};
#pragma unroll
        for (int a = 0; a < 2; ++a) {
          zd w[4];
#pragma unroll
          for (int X = 0; X < 4; ++X) {
            const zd w0 = S.W[X][ea[a] * N + f], w1 = S.W[X][ea[a] * N + f1];
            w[X] = pb0 * w0 + pb1 * w1;
            if (X == 3) cd += (a ? wr : -wr) * (w1 - w0);   // s_0 = -1, s_1 = +1
          }
          cw[0][a] = (h2 * wr) * w[0];
          cw[1][a] = (h2 * wr * k) * w[1];
          cw[2][a] = (h2 * wr) * (kt * w[2]);
          cw[3][a] = (-kk2h2 * wr) * w[3];
        }
      }
      for (int p = 0; p < q; ++p) {
        double row[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        if (ok) {
          const int64_t ip = e * q + p;
          const double xp = A.far.x[ip], yp = A.far.y[ip], nxp = A.far.nx[ip], nyp = A.far.ny[ip];
          const double u1 = A.wf[p] * A.xf[p], u0 = A.wf[p] - u1;
          const zd cS = u0 * cw[0][0] + u1 * cw[0][1];
          const zd cD = u0 * cw[1][0] + u1 * cw[1][1];      // times k
          const zd cT = u0 * cw[2][0] + u1 * cw[2][1];      // times k~
          const zd cN = u0 * cw[3][0] + u1 * cw[3][1];
          const double dx = xp - xq, dy = yp - yq;
          const double R2 = dx * dx + dy * dy, ri = rsqrt(R2), R = R2 * ri;
          const double ux = dx * ri, uy = dy * ri;
          const double g = ux * nxq + uy * nyq;
          const double nd = nxp * nxq + nyp * nyq;
          Hankel01 Hk, Ht;
          hankel_k_kt(A, R, Hk, Ht);
          const zd V = cD * Hk.H1 + cT * Ht.H1;              // dT/dn' along d^ (D, D~)
          const zd F0 = cT * Ht.H0, S1 = cS * Ht.H1, M0 = cN * Hk.H0;
          const zd un = ri * V;                              // dT/dd along n'
          // along d^: D and D~ g [kappa H0 - 2 H1 / R], S~ -k~ H1, N -k H1
          const zd uR = g * (k * (cD * Hk.H0) + kt * F0 - 2.0 * un) - kt * S1 -
                        k * ((A.wf[p] * cd + nd * cN) * Hk.H1);
          row[0] = uR.x * ux + un.x * nxq;
          row[1] = uR.y * ux + un.y * nxq;
          row[2] = uR.x * uy + un.x * nyq;
          row[3] = uR.y * uy + un.y * nyq;
          row[4] = M0.x * nxq;
          row[5] = M0.y * nxq;
          row[6] = M0.x * nyq;
          row[7] = M0.y * nyq;
#pragma unroll
          for (int i = 0; i < 4; ++i) col[i] -= row[i];
          col[4] += V.x * ux + M0.x * nxp;
          col[5] += V.y * ux + M0.y * nxp;
          col[6] += V.x * uy + M0.x * nyp;
          col[7] += V.y * uy + M0.y * nyp;
          // d/dk~: S~ and D~; the h^2-scaled part of T: all but the derivative part of N
          const zd dkt = R * (g * F0 - S1), val = cS * Ht.H0 + g * V + nd * M0;
          sc[0] += dkt.x; sc[1] += dkt.y; sc[2] += val.x; sc[3] += val.y;
        }
#pragma unroll
        for (int o = 16; o >= 4; o >>= 1) {
          const bool up = lane & o;
          const int m = o >> 2;   // 4, 2, 1 sums kept
#pragma unroll
          for (int i = 0; i < m; ++i) {
            const double send = up ? row[i] : row[i + m], keep = up ? row[i + m] : row[i];
            row[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
          }
        }
        row[0] += __shfl_xor_sync(0xffffffffu, row[0], 2);
        row[0] += __shfl_xor_sync(0xffffffffu, row[0], 1);
        if ((lane & 3) == 0) rowacc[warp][el][p][own] += row[0];
      }
    }
    if (fvalid) {
      double* gr = S.Gr + 4 * iq;
      double* gn = S.Gn + 4 * iq;
      // times i / 4
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        atomicAdd(gr + i, (i & 1) ? 0.25 * col[i - 1] : -0.25 * col[i + 1]);
        atomicAdd(gn + i, (i & 1) ? 0.25 * col[4 + i - 1] : -0.25 * col[4 + i + 1]);
      }
    }
  }
  // block sums of the scalars, then the row accumulators
#pragma unroll
  for (int i = 0; i < 4; ++i)
    for (int o = 16; o > 0; o >>= 1) sc[i] += __shfl_xor_sync(0xffffffffu, sc[i], o);
  if (lane == 0)
    for (int i = 0; i < 4; ++i) red[warp][i] = sc[i];
  __syncthreads();
  if (threadIdx.x < 4) {
    const int i = threadIdx.x;
    double t = 0.0;
    for (int w = 0; w < SH_W; ++w) t += red[w][i ^ 1];
    atomicAdd(S.scal + i, (i & 1) ? 0.25 * t : -0.25 * t);
  }
  for (int t = threadIdx.x; t < SH_E * q * 8; t += 32 * SH_W) {
    const int el = t / (q * 8), rem = t - el * q * 8, p = rem / 8, i = rem - p * 8;
    const int64_t e = e0 + el;
    double v = 0.0;
    for (int w = 0; w < SH_W; ++w) v += rowacc[w][el][p][i ^ 1];
    if (e < N) atomicAdd((i < 4 ? S.Gr : S.Gn) + 4 * (e * q + p) + (i & 3), (i & 1) ? 0.25 * v : -0.25 * v);
  }
}

// Near band: the W-weighted pair integrals of the element pairs with distance <=
// near_band, of two geometries at once (the two sides of a central difference), summed
// in a second kernel in the order (e, offset).  One warp per CTA and 32 pairs of one
// offset, so that the log-kernel pairs do not hold up warps of plain ones and the pairs
// spread over the whole GPU: one geometry with the offsets side by side ran 72 warps'
// quartets, each as long as its heaviest pairs (2 x 5.7 -> 3.9 ms at N = 1024).
// Where the recurrences' start depends on the warp (see band_sorts) the offsets stay
// side by side, whose grouping the FP64 values then follow.
__global__ void __launch_bounds__(32) k_shape_near(const __grid_constant__ AsmArgs A0, const __grid_constant__ AsmArgs A1,
                                                   const zd* W0, const zd* W1, const zd* W2, const zd* W3, zd* pairs,
                                                   int sorted) {
  const AsmArgs& A = blockIdx.y ? A1 : A0;
  const int64_t N = A.N, u = (int64_t)blockIdx.x * 32 + threadIdx.x;
  const int span = 2 * A.near_band + 1;
  int64_t e, off;
  if (sorted) {
    const int64_t nb = (N + 31) / 32;
    off = blockIdx.x / nb;
    e = u - off * nb * 32;
  } else {
    e = u / span;
    off = u - e * span;
  }
  if (e >= N) return;
  const int64_t f = ((e + off - A.near_band) % N + N) % N;
  zd acc = mkz(0.0);
  PairOut o;
  pair_integrals(A, e, f, o);
  const zd* W[4] = {W0, W1, W2, W3};
#pragma unroll
  for (int X = 0; X < 4; ++X)
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) acc += W[X][((e + a) % N) * N + (f + b) % N] * o.v[X][a * 2 + b];
  pairs[((int64_t)blockIdx.y * N + e) * span + off] = acc;
}

// block sums of n values each of the two geometries
__global__ void __launch_bounds__(128) k_shape_near_sum(const zd* pairs, int64_t n, double* part) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const zd acc = t < n ? pairs[blockIdx.y * n + t] : mkz(0.0);
  __shared__ double red[2][4];
  double v[2] = {acc.x, acc.y};
  for (int i = 0; i < 2; ++i)
    for (int o2 = 16; o2 > 0; o2 >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o2);
  if ((threadIdx.x & 31) == 0) { red[0][threadIdx.x >> 5] = v[0]; red[1][threadIdx.x >> 5] = v[1]; }
  __syncthreads();
  if (threadIdx.x == 0) {
    part += 2 * (int64_t)blockIdx.y * gridDim.x;
    part[2 * blockIdx.x] = red[0][0] + red[0][1] + red[0][2] + red[0][3];
    part[2 * blockIdx.x + 1] = red[1][0] + red[1][1] + red[1][2] + red[1][3];
  }
}

int shape_far_forms(const ShapeArgs& a, cudaStream_t s) {
  if (a.A.q_far > 16) { set_error("shape derivative: q_far <= 16"); return 1; }
  dim3 grid((unsigned)((a.A.N + SH_E - 1) / SH_E), (unsigned)((a.A.N + 32 * SH_W - 1) / (32 * SH_W)));
  k_shape_far<<<grid, 32 * SH_W, 0, s>>>(a);
  note_launch();
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) { set_error(std::string("shape (far): ") + cudaGetErrorString(err)); return 3; }
  return 0;
}

int shape_near_forms(const AsmArgs& A0, const AsmArgs& A1, const zd* const* W, zd* pairs, double* part, int* nparts,
                     cudaStream_t s) {
  const int64_t n = A0.N * (2 * A0.near_band + 1);
  const unsigned blocks = (unsigned)((n + 127) / 128);
  const bool sorted = band_sorts(A0) && band_sorts(A1);
  k_shape_near<<<dim3((unsigned)(sorted ? (A0.N + 31) / 32 * (2 * A0.near_band + 1) : (n + 31) / 32), 2), 32, 0, s>>>(
      A0, A1, W[0], W[1], W[2], W[3], pairs, sorted);
  note_launch();
  k_shape_near_sum<<<dim3(blocks, 2), 128, 0, s>>>(pairs, n, part);
  note_launch();
  *nparts = (int)blocks;
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) { set_error(std::string("shape (near): ") + cudaGetErrorString(err)); return 3; }
  return 0;
}

}  // namespace wcs
