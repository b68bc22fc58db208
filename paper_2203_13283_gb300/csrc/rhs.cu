// Plane-wave right-hand sides (Sec. II, Eq. 4) and the far-field map.
//
// exp(-i w t) convention; plane wave of propagation angle phi, d = (cos phi,
// sin phi), phase reference at the origin: H_z^inc = exp(i k d.r) and
// E_t^inc / eta = (d.n) exp(i k d.r).  [h]_i = int l_i H_z^inc,
// [e/eta]_i = int l_i E_t^inc / eta by q-point Gauss on the two elements of
// hat i.  Far field H^s ~ F(phi_o) e^{i k rho} / sqrt(rho),
// F = (i k e^{i pi/4} / sqrt(8 pi k)) int (x.n') e^{-i k x.r'} j ds'.
// Phases are formed and reduced in FP64 (k |r| reaches ~1e4).
#include "internal.h"

namespace wcs {

// Gauss rule on [0, 1], passed by value (no table shared between contexts, no
// synchronising upload per call)
struct Rule {
  double x[16], w[16];
};

__global__ void k_planewave(Rule R, Points P, int q, int64_t N, double h, double k, const double* angles,
                            int B, zd* e, zd* hv, int64_t ld) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int b = blockIdx.y;
  if (i >= N) return;
  double ds, dc;
  sincos(angles[b], &ds, &dc);
  zd se = mkz(0.0), sh = mkz(0.0);
  for (int a = 0; a < 2; ++a) {
    const int64_t el = (a == 1) ? (i - 1 + N) % N : i;  // a = 1: hat i is xi on element i-1
    for (int g = 0; g < q; ++g) {
      const int64_t ip = el * q + g;
      const double phi = (a == 1) ? R.x[g] : 1.0 - R.x[g];
      const double w = h * R.w[g] * phi;
      double s, c;
      sincos(k * (dc * P.x[ip] + ds * P.y[ip]), &s, &c);
      const double dn = dc * P.nx[ip] + ds * P.ny[ip];
      sh += mkz(w * c, w * s);
      se += mkz(w * dn * c, w * dn * s);
    }
  }
  e[(int64_t)b * ld + i] = se;
  hv[(int64_t)b * ld + i] = sh;
}

// Mixed form: the phase k d.r is split at a reference point r0 of hat i (its
// first Gauss point on element i): exp(i k d.r0) in FP64, once per angle, and
// exp(i k d.(r - r0)) in FP32, where |k d.(r - r0)| <= 2 k h stays small
// (~1e-7 absolute error).  A thread walks the 2q points of its hat once for
// PW_ANGLES angles.
constexpr int PW_ANGLES = 8;
__global__ void k_planewave_split(Rule R, Points P, int q, int64_t N, double h, double k, const double* angles,
                                  int B, zd* e, zd* hv, int64_t ld) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int b0 = blockIdx.y * PW_ANGLES;
  if (i >= N) return;
  const int nb = min(PW_ANGLES, B - b0);
  const double x0 = P.x[i * q], y0 = P.y[i * q];
  float dcf[PW_ANGLES], dsf[PW_ANGLES];
  float shr[PW_ANGLES], shi[PW_ANGLES], ser[PW_ANGLES], sei[PW_ANGLES];
#pragma unroll
  for (int a = 0; a < PW_ANGLES; ++a) {
    double sn = 0.0, cs = 1.0;
    if (a < nb) sincos(angles[b0 + a], &sn, &cs);
    dcf[a] = (float)cs;
    dsf[a] = (float)sn;
    shr[a] = shi[a] = ser[a] = sei[a] = 0.f;
  }
  const float kf = (float)k;
  for (int side = 0; side < 2; ++side) {
    const int64_t el = (side == 1) ? (i - 1 + N) % N : i;   // side 1: hat i is xi on element i-1
    for (int g = 0; g < q; ++g) {
      const int64_t ip = el * q + g;
      const float dx = (float)(P.x[ip] - x0), dy = (float)(P.y[ip] - y0);
      const float nx = (float)P.nx[ip], ny = (float)P.ny[ip];
      const float lam = (side == 1) ? (float)R.x[g] : (float)(1.0 - R.x[g]);
      const float w = (float)(h * R.w[g]) * lam;
#pragma unroll
      for (int a = 0; a < PW_ANGLES; ++a) {
        float sn, cs;
        sincosf(kf * (dcf[a] * dx + dsf[a] * dy), &sn, &cs);
        const float dn = w * (dcf[a] * nx + dsf[a] * ny);
        shr[a] = fmaf(w, cs, shr[a]);
        shi[a] = fmaf(w, sn, shi[a]);
        ser[a] = fmaf(dn, cs, ser[a]);
        sei[a] = fmaf(dn, sn, sei[a]);
      }
    }
  }
#pragma unroll
  for (int a = 0; a < PW_ANGLES; ++a) {
    if (a >= nb) break;
    double sn, cs;
    sincos(angles[b0 + a], &sn, &cs);
    double ps, pc;
    sincos(k * (cs * x0 + sn * y0), &ps, &pc);
    const zd ph = mkz(pc, ps);
    e[(int64_t)(b0 + a) * ld + i] = ph * mkz((double)ser[a], (double)sei[a]);
    hv[(int64_t)(b0 + a) * ld + i] = ph * mkz((double)shr[a], (double)shi[a]);
  }
}

__global__ void k_farfield_matrix(Rule R, Points P, int q, int64_t N, double h, double k, const double* phi,
                                  int nphi, zd* E, int64_t lde) {
  const int o = blockIdx.y;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  double os, oc;
  sincos(phi[o], &os, &oc);
  zd acc = mkz(0.0);
  for (int a = 0; a < 2; ++a) {
    const int64_t el = (a == 1) ? (i - 1 + N) % N : i;
    for (int g = 0; g < q; ++g) {
      const int64_t ip = el * q + g;
      const double lam = (a == 1) ? R.x[g] : 1.0 - R.x[g];
      const double w = h * R.w[g] * lam * (oc * P.nx[ip] + os * P.ny[ip]);
      double s, c;
      sincos(-k * (oc * P.x[ip] + os * P.y[ip]), &s, &c);
      acc += mkz(w * c, w * s);
    }
  }
  // i k e^{i pi/4} / sqrt(8 pi k)
  const double amp = k / sqrt(8.0 * WCS_PI * k);
  const zd pre = mkz(-amp * sqrt(0.5), amp * sqrt(0.5));
  E[i * lde + o] = pre * acc;
}

// The same map for the far field alone (k h <= 0.9; the shape gradient differences the
// map and keeps the kernel above).  There every node walks the 2 q points of its two
// elements, a full-range FP64 sincos each.  An element is short against the wavelength, so
// its part of the integral, as a function of the observation angle phi, is a short
// trigonometric polynomial: with d = k (y - y0) = r e^{i theta} from the element's middle
// point y0 (|r| < 0.55),
//   cos(r cos(phi - theta)) = J_0(r) + 2 sum_{even m} (-1)^(m/2) J_m(r) cos m(phi - theta),
//   sin(r cos(phi - theta)) = 2 sum_{odd m} (-1)^((m-1)/2) J_m(r) cos m(phi - theta)
// (Jacobi-Anger; terms above FM_M = 12 are below 4e-17), and the normal's factor moves
// each term by one harmonic.  k_farfield_moments sums the coefficients over the
// element's points once for all angles, one set for each of the element's two hats;
// k_farfield_map evaluates them: 56 FMA and one sincos per element and angle, whatever
// q, where walking the points with a Taylor polynomial each took 700 (5.6 ms at
// N = 16384, 360 angles).  Bound: FP64 pipe.
constexpr int FM_M = 12, FM_H = FM_M + 2;   // harmonics 0 .. FM_M + 1
constexpr int FM_NODES = 16;

// mom[(2 e + hat) FM_H + j] = H_j: the integral's cos part (odd j) and sin part (even j)
// are sums of Re(e^{i j phi} H_j).  Four lanes share the points of an element and hat.
__global__ void __launch_bounds__(128) k_farfield_moments(Rule R, Points P, int q, int64_t N, double h, double k, zd* mom) {
  const int64_t t = (int64_t)blockIdx.x * 128 + threadIdx.x;
  const int part = (int)(t & 3), hat = (int)((t >> 2) & 1);
  const bool ok = (t >> 3) < N;
  const int64_t e = ok ? t >> 3 : N - 1;
  const double* px = P.x + e * q;
  const double* py = P.y + e * q;
  const double x0 = px[q / 2], y0 = py[q / 2];
  zd H[FM_H];
#pragma unroll
  for (int j = 0; j < FM_H; ++j) H[j] = mkz(0.0);
  for (int g = part; g < q; g += 4) {
    const double w = h * R.w[g] * (hat ? R.x[g] : 1.0 - R.x[g]);
    const zd n = mkz(w * P.nx[e * q + g], w * P.ny[e * q + g]);
    const zd zeta = mkz(0.5 * k * (px[g] - x0), -0.5 * k * (py[g] - y0));
    const double s = abs2(zeta);
    // J_m(r) e^{-i m theta} = zeta^m / m! f_m, f_m = sum_i (-s)^i m! / (i! (m + i)!); the two
    // last by their series, the others by f_{m-1} = f_m - s f_{m+1} / (m (m + 1))
    double f[FM_M + 1], up = 1.0, fm = 1.0;
#pragma unroll
    for (int i = 7; i >= 1; --i) {
      up = fma(-s / (double)(i * (FM_M + 1 + i)), up, 1.0);
      fm = fma(-s / (double)(i * (FM_M + i)), fm, 1.0);
    }
    f[FM_M] = fm;
#pragma unroll
    for (int m = FM_M; m >= 1; --m) {
      const double lo = fma(-s * (1.0 / (double)(m * (m + 1))), up, f[m]);
      up = f[m];
      f[m - 1] = lo;
    }
    zd pw = mkz(1.0);
#pragma unroll
    for (int m = 0; m <= FM_M; ++m) {
      // half of the series' coefficient: cos m(phi - theta) times the normal's factor
      const double c = m == 0 ? f[0] : ((m / 2) % 2 ? -f[m] : f[m]);
      const zd G = c * pw;
      zfma(H[m + 1], conj(n), G);
      if (m >= 2) zfma(H[m - 1], n, G);
      if (m == 1) H[0].x += n.x * G.x - n.y * G.y;
      pw = (1.0 / (double)(m + 1)) * (pw * zeta);
    }
  }
#pragma unroll
  for (int j = 0; j < FM_H; ++j)
#pragma unroll
    for (int o = 1; o <= 2; o <<= 1) {
      H[j].x += __shfl_xor_sync(0xffffffffu, H[j].x, o);
      H[j].y += __shfl_xor_sync(0xffffffffu, H[j].y, o);
    }
  if (!ok || part) return;
#pragma unroll
  for (int j = 0; j < FM_H; ++j) mom[(2 * e + hat) * FM_H + j] = H[j];
}

// Lanes run over the observation angles (contiguous in the map); a thread walks FM_NODES
// elements and splits each element's integral between the hats of its two nodes.
__global__ void __launch_bounds__(128) k_farfield_map(const zd* __restrict__ mom, Points P, int q, int64_t N, double k,
                                                      const double* phi, int nphi, zd* E, int64_t lde) {
  const int o = blockIdx.x * 32 + (threadIdx.x & 31);
  const int64_t i0 = ((int64_t)blockIdx.y * 4 + (threadIdx.x >> 5)) * FM_NODES;
  if (o >= nphi || i0 >= N) return;
  double os, oc;
  sincos(phi[o], &os, &oc);
  double cj[FM_H], sj[FM_H];
  cj[0] = 1.0;
  sj[0] = 0.0;
#pragma unroll
  for (int j = 1; j < FM_H; ++j) {
    cj[j] = cj[j - 1] * oc - sj[j - 1] * os;
    sj[j] = cj[j - 1] * os + sj[j - 1] * oc;
  }
  const double amp = k / sqrt(8.0 * WCS_PI * k);
  const zd pre = mkz(-amp * sqrt(0.5), amp * sqrt(0.5));   // i k e^{i pi/4} / sqrt(8 pi k)
  const int64_t i1 = min(N, i0 + FM_NODES);
  zd right = mkz(0.0);   // of the element before the node: its share for the hat that rises on it
  for (int64_t i = i0 - 1; i < i1; ++i) {
    const int64_t e = i < 0 ? N - 1 : i;
    const zd* H = mom + 2 * e * FM_H;
    zd v[2];
#pragma unroll
    for (int hat = 0; hat < 2; ++hat) {
      double a = 0.0, b = H[hat * FM_H].x;
#pragma unroll
      for (int j = 1; j < FM_H; ++j) {
        const zd c = H[hat * FM_H + j];
        if (j & 1) a = fma(cj[j], c.x, fma(-sj[j], c.y, a));
        else b = fma(cj[j], c.x, fma(-sj[j], c.y, b));
      }
      v[hat] = mkz(a, -b);
    }
    double s0, c0;
    sincos(-k * fma(oc, P.x[e * q + q / 2], os * P.y[e * q + q / 2]), &s0, &c0);
    const zd ph = pre * mkz(c0, s0);
    if (i >= i0) E[i * lde + o] = ph * v[0] + right;
    right = ph * v[1];
  }
}

// Where the line lies: the moments cost ~100 us whatever the angles (one element's points are a
// chain of FP64 operations), more beyond 4000 elements, the points 1.7 ns an element and angle.
// Microseconds of a call, points / moments, one column: N = 1024 and 16, 64, 128 angles
// 153 / 248, 249 / 248, 341 / 250; N = 4096 and 8, 16, 32: 349 / 457, 412 / 455, 503 / 456;
// N = 16384 and 1, 16, 32: 264 / 684, 1371 / 1372, 1774 / 1371.
int64_t farfield_moments(int64_t N, int nphi, double kh) {
  const int64_t segs = (N + 4 * FM_NODES - 1) / (4 * FM_NODES);
  return nphi >= 16 && N * nphi >= 65536 && kh <= 0.9 && segs <= 65535 ? 2 * N * FM_H : 0;
}

static Rule rule(const double* xn, const double* wn, int q) {
  Rule R{};
  for (int i = 0; i < q; ++i) {
    R.x[i] = xn[i];
    R.w[i] = wn[i];
  }
  return R;
}

int planewave_rhs(const Points& near, const double* wn, const double* xn, int q, int64_t N,
                  double h, double k, const double* angles, int B, zd* e, zd* hv, int64_t ld,
                  cudaStream_t s, bool split_phase) {
  const Rule R = rule(xn, wn, q);
  if (split_phase) {
    for (int b0 = 0; b0 < B; b0 += 65535 * PW_ANGLES) {
      const int bb = std::min(65535 * PW_ANGLES, B - b0);
      dim3 g((unsigned)((N + 127) / 128), (unsigned)((bb + PW_ANGLES - 1) / PW_ANGLES));
      k_planewave_split<<<g, 128, 0, s>>>(R, near, q, N, h, k, angles + b0, bb, e + (int64_t)b0 * ld,
                                          hv + (int64_t)b0 * ld, ld);
      note_launch();
    }
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) { set_error(std::string("rhs: ") + cudaGetErrorString(err)); return 3; }
    return 0;
  }
  for (int b0 = 0; b0 < B; b0 += 65535) {
    int bb = std::min(65535, B - b0);
    dim3 g((unsigned)((N + 127) / 128), (unsigned)bb);
    k_planewave<<<g, 128, 0, s>>>(R, near, q, N, h, k, angles + b0, bb, e + (int64_t)b0 * ld,
                                  hv + (int64_t)b0 * ld, ld);
    note_launch();
  }
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) { set_error(std::string("rhs: ") + cudaGetErrorString(err)); return 3; }
  return 0;
}

int farfield_matrix(const Points& near, const double* wn, const double* xn, int q, int64_t N,
                    double h, double k, const double* phi, int nphi, zd* E, int64_t lde,
                    cudaStream_t s, zd* mom) {
  const Rule R = rule(xn, wn, q);
  if (mom) {
    const int64_t segs = (N + 4 * FM_NODES - 1) / (4 * FM_NODES);
    k_farfield_moments<<<(unsigned)((8 * N + 127) / 128), 128, 0, s>>>(R, near, q, N, h, k, mom);
    note_launch();
    k_farfield_map<<<dim3((unsigned)((nphi + 31) / 32), (unsigned)segs), 128, 0, s>>>(mom, near, q, N, k, phi, nphi, E, lde);
    note_launch();
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) { set_error(std::string("farfield: ") + cudaGetErrorString(err)); return 3; }
    return 0;
  }
  for (int o0 = 0; o0 < nphi; o0 += 65535) {
    int oo = std::min(65535, nphi - o0);
    dim3 g((unsigned)((N + 127) / 128), (unsigned)oo);
    k_farfield_matrix<<<g, 128, 0, s>>>(R, near, q, N, h, k, phi + o0, oo, E + o0, lde);
    note_launch();
  }
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) { set_error(std::string("farfield: ") + cudaGetErrorString(err)); return 3; }
  return 0;
}

}  // namespace wcs
