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

// The same map for the far field alone (k h <= 0.9; the shape gradient differences
// the map and keeps the kernel above).  There every node walks the 2 q points of
// its two elements, a full-range FP64 sincos each, and stores 16 bytes to a row of
// the column-major map.  Here lanes run over the observation angles (contiguous in
// the map), a thread walks FM_NODES elements and splits each element's integral
// between the hats of its two nodes as it goes; the phase is a sincos at the
// element's middle point and a Taylor polynomial of the difference, |d| <= k h < 0.9
// (to d^17 / d^16: omitted terms below 2e-17 / 1e-17 of 1 at 0.9, 1e-21 at 0.5).
// Bound: FP64 pipe, ~26 operations a point instead of ~80 twice.
constexpr int FM_NODES = 16;
__device__ __forceinline__ void cis_small(double d, double& s, double& c) {
  const double z = d * d;
  c = 4.779477332387385e-14;                     // 1 / 16!
  c = fma(c, z, -1.1470745597729725e-11);
  c = fma(c, z, 2.08767569878681e-09);
  c = fma(c, z, -2.755731922398589e-07);
  c = fma(c, z, 2.48015873015873e-05);
  c = fma(c, z, -0.001388888888888889);
  c = fma(c, z, 0.041666666666666664);
  c = fma(c, z, -0.5);
  c = fma(c, z, 1.0);
  s = 2.8114572543455206e-15;                    // 1 / 17!
  s = fma(s, z, -7.647163731819816e-13);
  s = fma(s, z, 1.6059043836821613e-10);
  s = fma(s, z, -2.505210838544172e-08);
  s = fma(s, z, 2.7557319223985893e-06);
  s = fma(s, z, -0.0001984126984126984);
  s = fma(s, z, 0.008333333333333333);
  s = fma(s, z, -0.16666666666666666);
  s = fma(s * z, d, d);
}

__global__ void __launch_bounds__(128) k_farfield_map(Rule R, Points P, int q, int64_t N, double h, double k, const double* phi,
                                                      int nphi, zd* E, int64_t lde) {
  const int o = blockIdx.x * 32 + (threadIdx.x & 31);
  const int64_t i0 = ((int64_t)blockIdx.y * 4 + (threadIdx.x >> 5)) * FM_NODES;
  if (o >= nphi || i0 >= N) return;
  double os, oc;
  sincos(phi[o], &os, &oc);
  const double amp = k / sqrt(8.0 * WCS_PI * k);
  const zd pre = mkz(-amp * sqrt(0.5), amp * sqrt(0.5));   // i k e^{i pi/4} / sqrt(8 pi k)
  const int64_t i1 = min(N, i0 + FM_NODES);
  zd right = mkz(0.0);   // of the element before the node: its share for the hat that rises on it
  for (int64_t i = i0 - 1; i < i1; ++i) {
    const int64_t e = i < 0 ? N - 1 : i;
    const double* px = P.x + e * q;
    const double* py = P.y + e * q;
    const double x0 = px[q / 2], y0 = py[q / 2];
    zd l = mkz(0.0), r = mkz(0.0);
    for (int g = 0; g < q; ++g) {
      const double d = -k * fma(oc, px[g] - x0, os * (py[g] - y0));
      double sn, cs;
      cis_small(d, sn, cs);
      const double w = h * R.w[g] * fma(oc, P.nx[e * q + g], os * P.ny[e * q + g]);
      const double wr = R.x[g] * w, wl = w - wr;
      l.x = fma(wl, cs, l.x);
      l.y = fma(wl, sn, l.y);
      r.x = fma(wr, cs, r.x);
      r.y = fma(wr, sn, r.y);
    }
    double s0, c0;
    sincos(-k * fma(oc, x0, os * y0), &s0, &c0);
    const zd ph = pre * mkz(c0, s0);
    if (i >= i0) E[i * lde + o] = ph * l + right;
    right = ph * r;
  }
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
                    cudaStream_t s, bool differenced) {
  const Rule R = rule(xn, wn, q);
  const int64_t segs = (N + 4 * FM_NODES - 1) / (4 * FM_NODES);
  if (!differenced && k * h <= 0.9 && segs <= 65535) {
    k_farfield_map<<<dim3((unsigned)((nphi + 31) / 32), (unsigned)segs), 128, 0, s>>>(R, near, q, N, h, k, phi, nphi, E, lde);
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
