// Staging of FP64 data into split-bf16 planes for the tensor-core contraction
// (split.cuh: x = p0 + p1 (+ p2), each plane the exact remainder rounded to
// nearest, formed with integer operations so that staging runs at memory
// speed rather than at GB300's FP64 rate).
#include <algorithm>

#include "gemm_tc.h"
#include "split.cuh"

namespace wcs {

__global__ void k_split_real(const double* X, int64_t rows, int64_t cols, int64_t ld, int planes,
                             uint16_t* p0, uint16_t* p1, uint16_t* p2, int64_t ldp) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t r = blockIdx.y;
  if (c >= cols) return;
  const int64_t o = r * ldp + c;
  uint16_t d1, d2;
  split3_bits(X[r * ld + c], planes, p0 + o, planes > 1 ? p1 + o : &d1, planes > 2 ? p2 + o : &d2);
}

int split_real_f64(const double* X, int64_t rows, int64_t cols, int64_t ld, int planes, uint16_t* const* P,
                   int64_t ldp, cudaStream_t s) {
  for (int64_t r0 = 0; r0 < rows; r0 += 65535) {
    const int64_t rr = std::min<int64_t>(65535, rows - r0);
    dim3 g((unsigned)((cols + 255) / 256), (unsigned)rr);
    k_split_real<<<g, 256, 0, s>>>(X + r0 * ld, rr, cols, ld, planes, P[0] + r0 * ldp,
                                   planes > 1 ? P[1] + r0 * ldp : nullptr, planes > 2 ? P[2] + r0 * ldp : nullptr, ldp);
    note_launch();
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { set_error(std::string("split: ") + cudaGetErrorString(e)); return 3; }
  return 0;
}

int split_complex_rows(const zd* X, int64_t rows, int64_t cols, int64_t ld, int planes, uint16_t* const* P,
                       int64_t ldp, cudaStream_t s) {
  return split_real_f64((const double*)X, rows, 2 * cols, 2 * ld, planes, P, ldp, s);
}

// One complex value of a right-hand block in the planes of B': row 2j: (Re x,
// -Im x), row 2j + 1: (Im x, Re x), each pair one 32-bit store (ldp and 2 i are
// even).  The planes of -v are those of v with the sign bits flipped.
__device__ __forceinline__ void stage_value(zd x, int planes, uint16_t* const (&P)[3], int64_t ldp, int64_t j, int64_t i) {
  uint16_t re[3] = {0, 0, 0}, im[3] = {0, 0, 0};
  split3_bits(x.x, planes, &re[0], &re[1], &re[2]);
  split3_bits(x.y, planes, &im[0], &im[1], &im[2]);
  const int64_t o0 = (2 * j) * ldp + 2 * i, o1 = o0 + ldp;
#pragma unroll
  for (int t = 0; t < 3; ++t) {
    if (t >= planes) break;
    *(uint32_t*)(P[t] + o0) = (uint32_t)re[t] | ((uint32_t)(im[t] ^ 0x8000u) << 16);
    *(uint32_t*)(P[t] + o1) = (uint32_t)im[t] | ((uint32_t)re[t] << 16);
  }
}

__global__ void k_stage_rhs(const zd* X, int64_t n, int64_t B, int64_t ldx, int conj_in, int planes,
                            uint16_t* p0, uint16_t* p1, uint16_t* p2, int64_t ldp) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t j = blockIdx.y;
  if (i >= n) return;
  zd x = X[j * ldx + i];
  if (conj_in) x.y = -x.y;
  uint16_t* const P[3] = {p0, p1, p2};
  stage_value(x, planes, P, ldp, j, i);
}

// y = G^-1 (x + ca a) + cz z for a segment of one column, with G^-1 as the forward
// and backward recursions of linalg.cu's Gram inverse, written as FP64 (y, optional)
// and as the staged planes of the next operator product.  One pass over memory
// replaces the vector update, both recursion passes and the staging pass (and the
// product G x / 2 inside the inverse, which is x / 2 outside it).  The segment and
// its margins lie in shared memory, 33 values a row so that the threads of the
// recursion, 32 values apart, meet no bank conflict.
// Bound: FP64 pipe, (32 + GS_WARM) / 32 x 4 FMAs a value, about the time of its
// 16 to 64 bytes of reads and 24 of planes.
constexpr int GS_SEG = 1024, GS_CH = 32, GS_WARM = 32, GS_THREADS = 128;   // |rho|^32 = 5e-19
constexpr int GS_LEN = GS_SEG + 2 * GS_WARM;
constexpr int GS_PAD = GS_LEN + GS_LEN / 32 + 1;
constexpr size_t GS_SMEM = 2 * sizeof(zd) * GS_PAD;

__device__ __forceinline__ int gs_at(int u) { return u + (u >> 5); }

__global__ void __launch_bounds__(GS_THREADS) k_gram_stage(GramStage g) {
  extern __shared__ zd gs[];
  zd* xs = gs;            // x, later the result
  zd* us = gs + GS_PAD;   // forward recursion
  const int64_t n = g.n, j = blockIdx.y, i0 = (int64_t)blockIdx.x * GS_SEG;
  const int len = (int)min((int64_t)GS_SEG, n - i0);
  const zd* x = g.x + j * g.ldx;
  const zd* add = g.add ? g.add + j * g.ld_add : nullptr;
  // margins: GS_WARM values on either side, cyclic
  for (int u = threadIdx.x; u < len + 2 * GS_WARM; u += GS_THREADS) {
    int64_t i = i0 + u - GS_WARM;
    if (i < 0 || i >= n) i = (i % n + n) % n;
    zd v = x[i];
    if (add) {
      const zd w = add[i];
      v.x = fma(g.ca.x, w.x, fma(-g.ca.y, w.y, v.x));
      v.y = fma(g.ca.x, w.y, fma(g.ca.y, w.x, v.y));
    }
    xs[gs_at(u)] = v;
  }
  __syncthreads();
  const double rho = g.rho;
  // forward over [GS_WARM, len + 2 GS_WARM), chunks of GS_CH
  for (int c = threadIdx.x; c * GS_CH < len + GS_WARM; c += GS_THREADS) {
    const int b = GS_WARM + c * GS_CH, e = min(b + GS_CH, len + 2 * GS_WARM);
    zd acc = mkz(0.0);
    for (int u = b - GS_WARM; u < b; ++u) acc = xs[gs_at(u)] + rho * acc;
    for (int u = b; u < e; ++u) {
      acc = xs[gs_at(u)] + rho * acc;
      us[gs_at(u)] = acc;
    }
  }
  __syncthreads();
  // backward over [GS_WARM, len + GS_WARM)
  for (int c = threadIdx.x; c * GS_CH < len; c += GS_THREADS) {
    const int b = GS_WARM + c * GS_CH, e = min(b + GS_CH, len + GS_WARM);
    zd acc = mkz(0.0);
    for (int u = e + GS_WARM - 1; u >= e; --u) acc = us[gs_at(u)] + rho * acc;
    for (int u = e - 1; u >= b; --u) {
      acc = us[gs_at(u)] + rho * acc;
      xs[gs_at(u)] = acc;
    }
  }
  __syncthreads();
  uint16_t* const P[3] = {g.P[0], g.P[1], g.P[2]};
  for (int u = threadIdx.x; u < len; u += GS_THREADS) {
    const int64_t i = i0 + u;
    zd v = g.scale * xs[gs_at(u + GS_WARM)];
    if (g.z) {
      const zd w = g.z[j * g.ldz + i];
      v.x = fma(g.cz, w.x, v.x);
      v.y = fma(g.cz, w.y, v.y);
    }
    if (g.y) g.y[j * g.ldy + i] = v;
    if (g.conj) v.y = -v.y;
    stage_value(v, g.planes, P, g.ldp, j, i);
  }
}

int gram_stage(GramStage g, int64_t cols, double h, cudaStream_t s) {
  if (cols <= 0) return 0;
  g.rho = sqrt(3.0) - 2.0;
  g.scale = -g.rho * 6.0 / h;
  static DeviceOnce attr;
  if (attr.need()) {
    cudaError_t e = cudaFuncSetAttribute(k_gram_stage, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GS_SMEM);
    if (e != cudaSuccess) { set_error(std::string("gram_stage: ") + cudaGetErrorString(e)); return 3; }
    attr.done();
  }
  for (int64_t c0 = 0; c0 < cols; c0 += 32768) {
    const int64_t cc = std::min<int64_t>(32768, cols - c0);
    GramStage q = g;
    q.x += c0 * g.ldx;
    if (g.add) q.add += c0 * g.ld_add;
    if (g.z) q.z += c0 * g.ldz;
    if (g.y) q.y += c0 * g.ldy;
    for (int p = 0; p < 3; ++p)
      if (g.P[p]) q.P[p] += 2 * c0 * g.ldp;
    dim3 grid((unsigned)((g.n + GS_SEG - 1) / GS_SEG), (unsigned)cc);
    k_gram_stage<<<grid, GS_THREADS, GS_SMEM, s>>>(q);
    note_launch();
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { set_error(std::string("gram_stage: ") + cudaGetErrorString(e)); return 3; }
  return 0;
}

// out = cb b + c1 (p + g G t), column by column (out may be p or b)
__global__ void k_gram_combine(const zd* p, int64_t ldp, const zd* __restrict__ t, int64_t ldt, double g6, double g4,
                               double c1, const zd* b, int64_t ldb, double cb, zd* out, int64_t ldo, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, c = blockIdx.y;
  if (i >= n) return;
  const zd* x = t + c * ldt;
  const zd m = x[i == 0 ? n - 1 : i - 1], x0 = x[i], q = x[i == n - 1 ? 0 : i + 1];
  zd r = p[c * ldp + i];
  r.x = fma(g4, x0.x, fma(g6, m.x + q.x, r.x));
  r.y = fma(g4, x0.y, fma(g6, m.y + q.y, r.y));
  r = c1 * r;
  if (b) {
    const zd w = b[c * ldb + i];
    r.x = fma(cb, w.x, r.x);
    r.y = fma(cb, w.y, r.y);
  }
  out[c * ldo + i] = r;
}

int gram_combine(const zd* p, int64_t ldp, const zd* t, int64_t ldt, double g, double c1, const zd* b, int64_t ldb,
                 double cb, zd* out, int64_t ldo, int64_t n, int64_t cols, double h, cudaStream_t s) {
  for (int64_t c0 = 0; c0 < cols; c0 += 65535) {
    const int64_t cc = std::min<int64_t>(65535, cols - c0);
    dim3 grid((unsigned)((n + 255) / 256), (unsigned)cc);
    k_gram_combine<<<grid, 256, 0, s>>>(p + c0 * ldp, ldp, t + c0 * ldt, ldt, g * h / 6.0, g * 4.0 * h / 6.0, c1,
                                        b ? b + c0 * ldb : nullptr, ldb, cb, out + c0 * ldo, ldo, n);
    note_launch();
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { set_error(std::string("gram_combine: ") + cudaGetErrorString(e)); return 3; }
  return 0;
}

int stage_rhs(const zd* X, int64_t n, int64_t B, int64_t ldx, int conj_in, int planes, uint16_t* const* P,
              int64_t ldp, cudaStream_t s) {
  for (int64_t b0 = 0; b0 < B; b0 += 32768) {
    const int64_t bb = std::min<int64_t>(32768, B - b0);
    dim3 g((unsigned)((n + 255) / 256), (unsigned)bb);
    k_stage_rhs<<<g, 256, 0, s>>>(X + b0 * ldx, n, bb, ldx, conj_in, planes, P[0] + 2 * b0 * ldp,
                                  planes > 1 ? P[1] + 2 * b0 * ldp : nullptr,
                                  planes > 2 ? P[2] + 2 * b0 * ldp : nullptr, ldp);
    note_launch();
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { set_error(std::string("stage_rhs: ") + cudaGetErrorString(e)); return 3; }
  return 0;
}

__global__ void k_stage_view(const zd* X, int64_t rows, int64_t cols, int64_t rs, int64_t cs, int conj,
                             int planes, uint16_t* p0, uint16_t* p1, uint16_t* p2, int64_t ldp) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t i = blockIdx.y;
  if (j >= cols) return;
  const zd x = X[i * rs + j * cs];
  // (Re x, Im x) adjacent: one 32-bit store per plane (ldp and 2 j are even)
  uint16_t re[3] = {0, 0, 0}, im[3] = {0, 0, 0};
  split3_bits(x.x, planes, &re[0], &re[1], &re[2]);
  split3_bits(conj ? -x.y : x.y, planes, &im[0], &im[1], &im[2]);
  uint16_t* P[3] = {p0, p1, p2};
  const int64_t o = i * ldp + 2 * j;
#pragma unroll
  for (int t = 0; t < 3; ++t) {
    if (t >= planes) break;
    *(uint32_t*)(P[t] + o) = (uint32_t)re[t] | ((uint32_t)im[t] << 16);
  }
}

int stage_view(const zd* X, int64_t rows, int64_t cols, int64_t rs, int64_t cs, int conj, int planes,
               uint16_t* const* P, int64_t ldp, cudaStream_t s) {
  for (int64_t r0 = 0; r0 < rows; r0 += 65535) {
    const int64_t rr = std::min<int64_t>(65535, rows - r0);
    dim3 g((unsigned)((cols + 255) / 256), (unsigned)rr);
    k_stage_view<<<g, 256, 0, s>>>(X + r0 * rs, rr, cols, rs, cs, conj, planes, P[0] + r0 * ldp,
                                   planes > 1 ? P[1] + r0 * ldp : nullptr, planes > 2 ? P[2] + r0 * ldp : nullptr,
                                   ldp);
    note_launch();
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { set_error(std::string("stage_view: ") + cudaGetErrorString(e)); return 3; }
  return 0;
}

}  // namespace wcs
