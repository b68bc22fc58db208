// Dense complex FP64 linear algebra for the solver: operator applies
// (Eq. 6), randomized range finding for the skeleton (Eq. 7) and the
// capacitance matrix of the Woodbury identity (Eq. 9).
#include <algorithm>
#include <climits>
#include <vector>

#include "internal.h"

namespace wcs {

// =========================================================================== ZGEMM (FP64 FMA pipe)
// C (m x n, column-major) = alpha * A * B + beta * C; A (m x k), B (k x n) are
// strided views (element (i, j) at p[i*rs + j*cs], optionally conjugated).
// 256 threads as a TY x TX grid, each computing TM x TN outputs: tiles of
// (TY TM) x (TX TN).  The FP64 pipe is the bound (GB300 issues ~2 DFMA per
// clock per SM), so the tile width follows n: a block of a few right-hand
// sides must not pay for 64 columns of zeros.
constexpr int GB_K = 16;

template <int TY, int TX, int TM, int TN>
__global__ void __launch_bounds__(256) k_zgemm(int64_t m, int64_t n, int64_t k, zd alpha, ZView A,
                                               ZView B, zd beta, zd* __restrict__ C, int64_t ldc) {
  static_assert(TY * TX == 256, "256 threads");
  constexpr int BM = TY * TM, BN = TX * TN;
  __shared__ zd As[GB_K][BM + 1];
  __shared__ zd Bs[GB_K][BN + 1];
  const int tx = threadIdx.x % TX, ty = threadIdx.x / TX;
  const int64_t m0 = (int64_t)blockIdx.y * BM, n0 = (int64_t)blockIdx.x * BN;
  zd acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = mkz(0.0);
  const bool a_kfast = (A.cs == 1);  // walk k first when it is the contiguous index
  const bool b_kfast = (B.rs == 1);
  for (int64_t k0 = 0; k0 < k; k0 += GB_K) {
    for (int u = threadIdx.x; u < BM * GB_K; u += 256) {
      int ii, kk;
      if (a_kfast) { kk = u % GB_K; ii = u / GB_K; } else { ii = u % BM; kk = u / BM; }
      const int64_t gi = m0 + ii, gk = k0 + kk;
      zd v = mkz(0.0);
      if (gi < m && gk < k) {
        v = A.p[gi * A.rs + gk * A.cs];
        if (A.conj) v.y = -v.y;
      }
      As[kk][ii] = v;
    }
    for (int u = threadIdx.x; u < BN * GB_K; u += 256) {
      int jj, kk;
      if (b_kfast) { kk = u % GB_K; jj = u / GB_K; } else { jj = u % BN; kk = u / BN; }
      const int64_t gj = n0 + jj, gk = k0 + kk;
      zd v = mkz(0.0);
      if (gj < n && gk < k) {
        v = B.p[gk * B.rs + gj * B.cs];
        if (B.conj) v.y = -v.y;
      }
      Bs[kk][jj] = v;
    }
    __syncthreads();
#pragma unroll 4
    for (int kk = 0; kk < GB_K; ++kk) {
      zd a[TM], b[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = As[kk][ty + TY * i];
#pragma unroll
      for (int j = 0; j < TN; ++j) b[j] = Bs[kk][tx + TX * j];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) zfma(acc[i][j], a[i], b[j]);
    }
    __syncthreads();
  }
  const bool beta0 = (beta.x == 0.0 && beta.y == 0.0);
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int64_t gi = m0 + ty + TY * i, gj = n0 + tx + TX * j;
      if (gi < m && gj < n) {
        zd r = alpha * acc[i][j];
        if (!beta0) r += beta * C[gj * ldc + gi];
        C[gj * ldc + gi] = r;
      }
    }
}

template <int TY, int TX, int TM, int TN>
static int launch_zgemm(int64_t m, int64_t n, int64_t k, zd alpha, ZView A, ZView B, zd beta, zd* C, int64_t ldc,
                        cudaStream_t s) {
  constexpr int BM = TY * TM, BN = TX * TN;
  dim3 grid((unsigned)((n + BN - 1) / BN), (unsigned)((m + BM - 1) / BM));
  if (grid.y > 65535) { set_error("zgemm: m too large"); return 1; }
  k_zgemm<TY, TX, TM, TN><<<grid, 256, 0, s>>>(m, n, k, alpha, A, B, beta, C, ldc);
  note_launch();
  return 0;
}

// Products too small to fill the GPU with output tiles: the K loop is spread
// over the lanes (or the warps) of a CTA instead, so that the 256 x 256
// product of one plane wave runs on hundreds of warps rather than on two CTAs
// of a serial K loop (N = 256, one column: 300 us in k_zgemm, 4.7 us here).
// What bounds them is the FP64 pipe for 4 and more columns, the latency of
// one pass over A below that.  Sums are formed in a fixed order.
//
// k_zgemm_rows: K contiguous in A (A.cs == 1): one warp per row, lanes over K,
// NC columns per pass, shuffle reduction.
template <int NC>
__global__ void __launch_bounds__(128) k_zgemm_rows(int64_t m, int64_t n, int64_t k, zd alpha, ZView A, ZView B,
                                                    zd beta, zd* __restrict__ C, int64_t ldc) {
  const int lane = threadIdx.x & 31;
  const int64_t i = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5), j0 = (int64_t)blockIdx.y * NC;
  if (i >= m) return;
  zd acc[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) acc[c] = mkz(0.0);
  const zd* a = A.p + i * A.rs;
#pragma unroll 2
  for (int64_t t = lane; t < k; t += 32) {
    zd v = a[t];
    if (A.conj) v.y = -v.y;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      if (j0 + c < n) {
        zd w = B.p[t * B.rs + (j0 + c) * B.cs];
        if (B.conj) w.y = -w.y;
        zfma(acc[c], v, w);
      }
    }
  }
#pragma unroll
  for (int c = 0; c < NC; ++c)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      acc[c].x += __shfl_xor_sync(0xffffffffu, acc[c].x, o);
      acc[c].y += __shfl_xor_sync(0xffffffffu, acc[c].y, o);
    }
  // lane c stores column c
  zd r = acc[0];
#pragma unroll
  for (int c = 1; c < NC; ++c)
    if (lane == c) r = acc[c];
  if (lane < NC && j0 + lane < n) {
    zd* o = C + (j0 + lane) * ldc + i;
    r = alpha * r;
    if (!(beta.x == 0.0 && beta.y == 0.0)) r += beta * (*o);
    *o = r;
  }
}

// k_zgemm_cols: rows contiguous in A (A.rs == 1): lanes over 32 rows, the 16
// warps of a CTA over K, their sums joined through shared memory in order.
template <int NC>
__global__ void __launch_bounds__(512) k_zgemm_cols(int64_t m, int64_t n, int64_t k, zd alpha, ZView A, ZView B,
                                                    zd beta, zd* __restrict__ C, int64_t ldc) {
  __shared__ zd part[16][NC][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t i = (int64_t)blockIdx.x * 32 + lane, j0 = (int64_t)blockIdx.y * NC;
  zd acc[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) acc[c] = mkz(0.0);
  if (i < m) {
#pragma unroll 2
    for (int64_t t = warp; t < k; t += 16) {
      zd v = A.p[i + t * A.cs];
      if (A.conj) v.y = -v.y;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        if (j0 + c < n) {
          zd w = B.p[t * B.rs + (j0 + c) * B.cs];
          if (B.conj) w.y = -w.y;
          zfma(acc[c], v, w);
        }
      }
    }
  }
#pragma unroll
  for (int c = 0; c < NC; ++c) part[warp][c][lane] = acc[c];
  __syncthreads();
  for (int c = warp; c < NC; c += 16) {
    zd r = part[0][c][lane];
#pragma unroll
    for (int w = 1; w < 16; ++w) r += part[w][c][lane];
    if (i < m && j0 + c < n) {
      zd* o = C + (j0 + c) * ldc + i;
      r = alpha * r;
      if (!(beta.x == 0.0 && beta.y == 0.0)) r += beta * (*o);
      *o = r;
    }
  }
}

template <int NC>
static void launch_zgemm_small(bool rows, int64_t m, int64_t n, int64_t k, zd alpha, ZView A, ZView B, zd beta, zd* C,
                               int64_t ldc, cudaStream_t s) {
  if (rows) {
    dim3 g((unsigned)((m + 3) / 4), (unsigned)((n + NC - 1) / NC));
    k_zgemm_rows<NC><<<g, 128, 0, s>>>(m, n, k, alpha, A, B, beta, C, ldc);
  } else {
    dim3 g((unsigned)((m + 31) / 32), (unsigned)((n + NC - 1) / NC));
    k_zgemm_cols<NC><<<g, 512, 0, s>>>(m, n, k, alpha, A, B, beta, C, ldc);
  }
  note_launch();
}

// The spread kernels serve up to 8 columns of any length (every column pass
// reads A once) and wider products of up to 2^22 complex multiply-adds, for
// which the tile kernel has too few tiles (64 x 64 x 64: one CTA).  Columns
// per pass: the most that leaves about two CTAs per SM.
static bool zgemm_small(int64_t m, int64_t n, int64_t k, zd alpha, ZView A, ZView B, zd beta, zd* C, int64_t ldc,
                        cudaStream_t s) {
  const bool rows = (A.cs == 1);
  if (!rows && A.rs != 1) return false;
  if (n > 8 && (double)m * (double)n * (double)k > 4194304.0) return false;
  if (n > 65535) return false;
  const int64_t tiles = rows ? (m + 3) / 4 : (m + 31) / 32;
  int nc = 8;
  while (nc > 1 && (nc / 2 >= n || tiles * ((n + nc - 1) / nc) < 304)) nc /= 2;
  switch (nc) {
    case 8: launch_zgemm_small<8>(rows, m, n, k, alpha, A, B, beta, C, ldc, s); break;
    case 4: launch_zgemm_small<4>(rows, m, n, k, alpha, A, B, beta, C, ldc, s); break;
    case 2: launch_zgemm_small<2>(rows, m, n, k, alpha, A, B, beta, C, ldc, s); break;
    default: launch_zgemm_small<1>(rows, m, n, k, alpha, A, B, beta, C, ldc, s); break;
  }
  return true;
}

// K in order, for up to eight columns: a half-warp's 16 lanes form the real and
// the other 16 the imaginary parts of 16 rows of one column, with the operations
// of zfma in k_zgemm's order (the same bits).  Bound by the FP64 pipe, whose
// quarter of an SM issues one warp instruction in 64 clocks: 2 K of them a warp
// (63 us at K = 1024).  Operand tiles of ZS_K steps come through shared memory, ZS_ST in
// flight: with plain loads the chain waited for them (410 us, cold caches).
constexpr int ZS_K = 32, ZS_ST = 4;
__global__ void __launch_bounds__(128) k_zgemm_serial(int64_t m, int64_t n, int64_t k, zd alpha, ZView A, ZView B,
                                                      zd beta, zd* __restrict__ C, int64_t ldc) {
  __shared__ zd as[ZS_ST][16][ZS_K + 1], bs[ZS_ST][4][ZS_K + 1];
  const int tid = threadIdx.x, lane = tid & 31, half = lane >> 4, warp = tid >> 5;
  const int64_t i0 = (int64_t)blockIdx.x * 16, j0 = (int64_t)blockIdx.y * 4;
  const int64_t tiles = (k + ZS_K - 1) / ZS_K;
  auto copy = [](zd* dst, const zd* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
  };
  auto fetch = [&](int64_t t) {
    if (t < tiles) {
      const int st = (int)(t % ZS_ST);
      const int64_t k0 = t * ZS_K;
#pragma unroll
      for (int u = tid; u < 16 * ZS_K; u += 128) {   // lanes along the operand's contiguous index
        const int r = A.cs == 1 ? u / ZS_K : u % 16, c = A.cs == 1 ? u % ZS_K : u / 16;
        if (k0 + c < k) copy(&as[st][r][c], A.p + min(i0 + r, m - 1) * A.rs + (k0 + c) * A.cs);
      }
      const int r = B.cs == 1 ? tid % 4 : tid / ZS_K, c = B.cs == 1 ? tid / 4 : tid % ZS_K;
      if (k0 + c < k) copy(&bs[st][r][c], B.p + min(j0 + r, n - 1) * B.cs + (k0 + c) * B.rs);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");   // one group per tile, also past the last
  };
  for (int t = 0; t < ZS_ST - 1; ++t) fetch(t);
  double acc = 0.0;
  for (int64_t t = 0; t < tiles; ++t) {
    asm volatile("cp.async.wait_group %0;" ::"n"(ZS_ST - 2) : "memory");
    __syncthreads();               // tile t is there; tile t - 1's stage is free
    fetch(t + ZS_ST - 1);
    const zd* a = as[t % ZS_ST][lane & 15];
    const zd* b = bs[t % ZS_ST][warp];
    const int steps = (int)min((int64_t)ZS_K, k - t * ZS_K);
#pragma unroll 8
    for (int c = 0; c < steps; ++c) {
      zd v = a[c], w = b[c];
      if (A.conj) v.y = -v.y;
      if (B.conj) w.y = -w.y;
      // re: fma(a.x, b.x, fma(-a.y, b.y, re)); im: fma(a.x, b.y, fma(a.y, b.x, im))
      acc = fma(v.x, half ? w.y : w.x, fma(half ? v.y : -v.y, half ? w.x : w.y, acc));
    }
  }
  const double im = __shfl_down_sync(0xffffffffu, acc, 16);
  const int64_t i = i0 + (lane & 15), j = j0 + warp;
  if (half || i >= m || j >= n) return;
  zd r = alpha * mkz(acc, im);
  zd* o = C + j * ldc + i;
  if (!(beta.x == 0.0 && beta.y == 0.0)) r += beta * (*o);
  *o = r;
}

// Every tile shape sums an entry over k in the same order, so the tile follows
// the shape: the largest that still gives two CTAs per SM (N = 1024, 32
// columns: 16 CTAs of 64 x 64 tiles took 1.2 ms, 128 of 16 x 16 take 0.2).
int zgemm_ordered(int64_t m, int64_t n, int64_t k, zd alpha, ZView A, ZView B, zd beta, zd* C, int64_t ldc,
                  cudaStream_t s) {
  if (m <= 0 || n <= 0) return 0;
  int r = 0;
  auto tiles = [&](int64_t t) { return ((m + t - 1) / t) * ((n + t - 1) / t); };
  if (n <= 8) {
    dim3 g((unsigned)((m + 15) / 16), (unsigned)((n + 3) / 4));
    k_zgemm_serial<<<g, 128, 0, s>>>(m, n, k, alpha, A, B, beta, C, ldc);
    note_launch();
  } else if (tiles(64) >= 304 || m > 65535 * 32) {
    r = launch_zgemm<16, 16, 4, 4>(m, n, k, alpha, A, B, beta, C, ldc, s);   // 64 x 64
  } else if (tiles(32) >= 304 || m > 65535 * 16) {
    r = launch_zgemm<16, 16, 2, 2>(m, n, k, alpha, A, B, beta, C, ldc, s);   // 32 x 32
  } else {
    r = launch_zgemm<16, 16, 1, 1>(m, n, k, alpha, A, B, beta, C, ldc, s);   // 16 x 16
  }
  if (r) return r;
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) { set_error(std::string("zgemm: ") + cudaGetErrorString(err)); return 3; }
  return 0;
}

int zgemm(int64_t m, int64_t n, int64_t k, zd alpha, ZView A, ZView B, zd beta, zd* C, int64_t ldc,
          cudaStream_t s) {
  if (m <= 0 || n <= 0) return 0;
  if (!zgemm_small(m, n, k, alpha, A, B, beta, C, ldc, s)) return zgemm_ordered(m, n, k, alpha, A, B, beta, C, ldc, s);
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) { set_error(std::string("zgemm: ") + cudaGetErrorString(err)); return 3; }
  return 0;
}

// =========================================================================== Gram matrix
// G = (h/6) circ(1, 4, 1).  With rho = sqrt(3) - 2 (root of rho^2 + 4 rho + 1):
// circ(1,4,1) = (-1/rho) (1 - rho S)(1 - rho S^-1), S the cyclic down-shift,
// so G^{-1} x = (6/h)(-rho) z with u_i = x_i + rho u_{i-1} (forward) and
// z_i = u_i + rho z_{i+1} (backward).  Each thread filters a chunk of CH
// outputs starting WARM samples early; |rho|^WARM < 1e-23 makes the cyclic
// wrap-around exact to rounding.
constexpr int GI_CH = 64, GI_WARM = 40;

__global__ void k_gram_fwd(const zd* __restrict__ X, int64_t ldx, zd* __restrict__ U, int64_t n,
                           int64_t cols, double rho) {
  const int64_t chunks = (n + GI_CH - 1) / GI_CH;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= chunks * cols) return;
  const int64_t c = t / chunks, i0 = (t - c * chunks) * GI_CH;
  const int64_t i1 = min(n, i0 + GI_CH);
  const zd* x = X + c * ldx;
  zd* u = U + c * n;
  zd acc = mkz(0.0);
  const int64_t warm = GI_WARM;  // the input is periodic: wrapping more than once is fine
  int64_t ii = ((i0 - warm) % n + n) % n;   // index mod n, advanced with a compare (no division per step)
  for (int64_t i = i0 - warm; i < i1; ++i) {
    acc = x[ii] + rho * acc;
    if (i >= i0) u[ii] = acc;
    if (++ii == n) ii = 0;
  }
}

__global__ void k_gram_bwd(const zd* __restrict__ U, zd* __restrict__ Y, int64_t ldy, int64_t n,
                           int64_t cols, double rho, double scale) {
  const int64_t chunks = (n + GI_CH - 1) / GI_CH;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= chunks * cols) return;
  const int64_t c = t / chunks, i0 = (t - c * chunks) * GI_CH;
  const int64_t i1 = min(n, i0 + GI_CH);
  const zd* u = U + c * n;
  zd* y = Y + c * ldy;
  zd acc = mkz(0.0);
  const int64_t warm = GI_WARM;
  int64_t ii = (i1 - 1 + warm) % n;
  for (int64_t i = i1 - 1 + warm; i >= i0; --i) {
    acc = u[ii] + rho * acc;
    if (i < i1) y[ii] = scale * acc;
    if (--ii < 0) ii = n - 1;
  }
}

// Both filters in one kernel, the same values.  The kernels above walk a chunk with one
// thread, every sample a load from memory behind the last (45 us for one column of 256,
// where the two chains of 104 dependent FMA take 7).  Here a CTA keeps up to GI_SLOTS
// chunks of one column in shared memory, each with its own GI_WARM samples before it, and
// two lanes (real and imaginary part) filter each chunk in place.  A chunk's backward
// filter starts in the next one, behind a short last chunk in the one after it: with more
// than GI_SLOTS chunks a CTA also runs the forward filter of the two that follow its own.
constexpr int GI_SLOTS = 32, GI_LD = GI_CH + GI_WARM + 1;   // odd stride: no bank conflicts
constexpr int64_t GI_FUSED_CHUNKS = 16384, GI_FUSED_CTAS = 2560;

__global__ void __launch_bounds__(2 * GI_SLOTS) k_gram_inverse(const zd* X, int64_t ldx, zd* Y, int64_t ldy, int64_t n,
                                                               int per, double rho, double scale) {
  extern __shared__ zd gi[];
  const int64_t chunks = (n + GI_CH - 1) / GI_CH, c0 = (int64_t)blockIdx.y * per;
  const int own = (int)min((int64_t)per, chunks - c0);
  const bool ring = chunks <= GI_SLOTS;
  const int slots = ring ? own : own + 2;
  const int last = (int)(n - (chunks - 1) * GI_CH);   // samples of the last chunk
  const zd* x = X + (int64_t)blockIdx.x * ldx;
  auto chunk = [&](int q) { return c0 + q < chunks ? c0 + q : c0 + q - chunks; };
  auto len = [&](int q) { return chunk(q) == chunks - 1 ? last : GI_CH; };
  for (int u = threadIdx.x; u < slots * (GI_CH + GI_WARM); u += blockDim.x) {
    const int q = u / (GI_CH + GI_WARM), t = u - q * (GI_CH + GI_WARM);
    if (t >= GI_WARM + len(q)) continue;
    int64_t ii = chunk(q) * GI_CH + t - GI_WARM;
    while (ii < 0) ii += n;
    gi[q * GI_LD + t] = x[ii];
  }
  __syncthreads();
  const int q = threadIdx.x >> 1;
  double* g = (double*)gi + (threadIdx.x & 1);
  if (q < slots) {
    double acc = 0.0, *p = g + 2 * q * GI_LD;
    const int m = len(q);
#pragma unroll 8
    for (int t = 0; t < GI_WARM; ++t) acc = fma(rho, acc, p[2 * t]);
    p += 2 * GI_WARM;
#pragma unroll 8
    for (int t = 0; t < m; ++t) {
      acc = fma(rho, acc, p[2 * t]);
      p[2 * t] = acc;
    }
  }
  __syncthreads();
  double acc = 0.0;
  if (q < own) {
    int cur = q, off = len(q) - 1 + GI_WARM;
    while (off >= len(cur)) {
      off -= len(cur);
      cur = (ring && cur + 1 == own) ? 0 : cur + 1;
    }
#pragma unroll 4
    for (int t = 0; t < GI_WARM; ++t) {
      acc = fma(rho, acc, g[2 * (cur * GI_LD + GI_WARM + off)]);
      if (--off < 0) {
        cur = (ring && cur == 0) ? own - 1 : cur - 1;
        off = len(cur) - 1;
      }
    }
  }
  __syncthreads();   // the filters write in place from here on
  if (q < own) {
    double* p = g + 2 * (q * GI_LD + GI_WARM);
#pragma unroll 8
    for (int t = len(q) - 1; t >= 0; --t) {
      acc = fma(rho, acc, p[2 * t]);
      p[2 * t] = scale * acc;
    }
  }
  __syncthreads();
  zd* y = Y + (int64_t)blockIdx.x * ldy + c0 * GI_CH;
  for (int u = threadIdx.x; u < own * GI_CH; u += blockDim.x) {
    const int b = u / GI_CH, t = u - b * GI_CH;
    if (t < len(b)) y[u] = gi[b * GI_LD + GI_WARM + t];
  }
}

int gram_inverse(const zd* X, int64_t ldx, zd* Y, int64_t ldy, int64_t n, int64_t cols, double h,
                 zd* work, cudaStream_t s) {
  if (cols <= 0) return 0;
  if (!work) { set_error("gram: no work buffer"); return 1; }
  const double rho = sqrt(3.0) - 2.0;
  const int64_t chunks = (n + GI_CH - 1) / GI_CH;
  const bool apart = Y + (cols - 1) * ldy + n <= X || X + (cols - 1) * ldx + n <= Y;
  const int per = chunks <= GI_SLOTS ? (int)chunks : GI_SLOTS - 2;
  const int64_t ctas = cols * ((chunks + per - 1) / per);
  // One kernel while its CTAs, four to an SM for their shared memory, go round few times;
  // the two passes where all their chains run at once anyway.  us for both, N = 2777:
  // 42 and 64 at 12288 chunks, 55 and 62 at 16384, 70 and 72 at 24576, 177 and 136 at
  // 65536; N = 32768: 46 and 62, 78 and 72 at 24576, 674 and 473 at 262144.  Columns of few
  // chunks leave lanes idle, so the CTAs count too: N = 64, 40 and 57 at 2048, 72 and 57 at
  // 4096, 525 and 72 at 32768; N = 200, 42 and 59 at 2048, 60 and 59 at 3072.
  // In place only where one CTA holds the whole column.
  if (chunks * cols <= GI_FUSED_CHUNKS && ctas <= GI_FUSED_CTAS && (chunks <= GI_SLOTS || apart)) {
    const size_t smem = sizeof(zd) * GI_LD * (chunks <= GI_SLOTS ? chunks : GI_SLOTS);
    static DeviceOnce attr;
    if (attr.need()) {
      cudaError_t e = cudaFuncSetAttribute(k_gram_inverse, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)(sizeof(zd) * GI_LD * GI_SLOTS));
      if (e != cudaSuccess) { set_error(std::string("gram: ") + cudaGetErrorString(e)); return 3; }
      attr.done();
    }
    k_gram_inverse<<<dim3((unsigned)cols, (unsigned)(ctas / cols)), 2 * GI_SLOTS, smem, s>>>(
        X, ldx, Y, ldy, n, per, rho, -rho * 6.0 / h);
    note_launch();
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) { set_error(std::string("gram: ") + cudaGetErrorString(err)); return 3; }
    return 0;
  }
  const int64_t tasks = ((n + GI_CH - 1) / GI_CH) * cols;
  const unsigned blocks = (unsigned)((tasks + 127) / 128);
  k_gram_fwd<<<blocks, 128, 0, s>>>(X, ldx, work, n, cols, rho);
  note_launch();
  k_gram_bwd<<<blocks, 128, 0, s>>>(work, Y, ldy, n, cols, rho, -rho * 6.0 / h);
  note_launch();
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) { set_error(std::string("gram: ") + cudaGetErrorString(err)); return 3; }
  return 0;
}

__global__ void k_gram_apply(const zd* __restrict__ X, int64_t ldx, zd* __restrict__ Y, int64_t ldy,
                             int64_t n, double a6, double a4, double beta) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t c = blockIdx.y;
  if (i >= n) return;
  const zd* x = X + c * ldx;
  const zd xm = x[i == 0 ? n - 1 : i - 1], x0 = x[i], xp = x[i == n - 1 ? 0 : i + 1];
  zd r = a6 * (xm + xp) + a4 * x0;
  zd* y = Y + c * ldy;
  if (beta != 0.0) r += beta * y[i];
  y[i] = r;
}

int gram_apply(const zd* X, int64_t ldx, zd* Y, int64_t ldy, int64_t n, int64_t cols, double h,
               double alpha, double beta, cudaStream_t s) {
  for (int64_t c0 = 0; c0 < cols; c0 += 65535) {
    int64_t cc = std::min<int64_t>(65535, cols - c0);
    dim3 g((unsigned)((n + 255) / 256), (unsigned)cc);
    k_gram_apply<<<g, 256, 0, s>>>(X + c0 * ldx, ldx, Y + c0 * ldy, ldy, n, alpha * h / 6.0,
                                   alpha * 4.0 * h / 6.0, beta);
    note_launch();
  }
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) { set_error(std::string("gram_apply: ") + cudaGetErrorString(err)); return 3; }
  return 0;
}

// =========================================================================== small kernels
__global__ void k_colnorm(const zd* X, int64_t ld, int64_t m, double* out) {
  __shared__ double red[256];
  const int64_t c = blockIdx.x;
  double s = 0.0;
  for (int64_t i = threadIdx.x; i < m; i += blockDim.x) s += abs2(X[c * ld + i]);
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[c] = sqrt(red[0]);
}

__global__ void k_coldotc(const zd* X, int64_t ldx, const zd* Y, int64_t ldy, int64_t m, zd* out) {
  __shared__ double re[256], im[256];
  const int64_t c = blockIdx.x;
  zd s = mkz(0.0);
  for (int64_t i = threadIdx.x; i < m; i += blockDim.x) s += conj(X[c * ldx + i]) * Y[c * ldy + i];
  re[threadIdx.x] = s.x;
  im[threadIdx.x] = s.y;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      re[threadIdx.x] += re[threadIdx.x + o];
      im[threadIdx.x] += im[threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) out[c] = mkz(re[0], im[0]);
}

int column_dotc(const zd* X, int64_t ldx, const zd* Y, int64_t ldy, int64_t m, int64_t n, zd* out,
                cudaStream_t s) {
  for (int64_t c0 = 0; c0 < n; c0 += 65535) {
    const int64_t cc = std::min<int64_t>(65535, n - c0);
    k_coldotc<<<(unsigned)cc, 256, 0, s>>>(X + c0 * ldx, ldx, Y + c0 * ldy, ldy, m, out + c0);
    note_launch();
  }
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) { set_error(cudaGetErrorString(err)); return 3; }
  return 0;
}

int column_norms(const zd* X, int64_t ld, int64_t m, int64_t n, double* out, cudaStream_t s) {
  if (n <= 0) return 0;
  k_colnorm<<<(unsigned)n, 256, 0, s>>>(X, ld, m, out);
  note_launch();
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) { set_error(cudaGetErrorString(err)); return 3; }
  return 0;
}

// Philox-4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11)
__device__ __forceinline__ uint4 philox4x32(uint4 c, uint2 k) {
  const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u, W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t hi0 = __umulhi(M0, c.x), lo0 = M0 * c.x;
    const uint32_t hi1 = __umulhi(M1, c.z), lo1 = M1 * c.z;
    c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
    k.x += W0;
    k.y += W1;
  }
  return c;
}

__device__ __forceinline__ double u01(uint32_t a, uint32_t b) {
  // 53-bit uniform in (0, 1]
  const uint64_t v = ((uint64_t)a << 21) ^ (uint64_t)b;
  return ((double)(v & ((1ull << 53) - 1)) + 1.0) * (1.0 / 9007199254740992.0);
}

__global__ void k_gauss(zd* X, int64_t ld, int64_t m, int64_t n, uint64_t seed, uint64_t offset) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= m * n) return;
  const int64_t c = t / m, i = t - c * m;
  const uint64_t ctr = offset + (uint64_t)t;
  uint4 r = philox4x32(make_uint4((uint32_t)ctr, (uint32_t)(ctr >> 32), 0x57435331u, 0u),
                       make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
  const double u1 = u01(r.x, r.y), u2 = u01(r.z, r.w);
  const double rad = sqrt(-log(u1));  // E|z|^2 = 1
  double sn, cs;
  sincospi(2.0 * u2, &sn, &cs);
  X[c * ld + i] = mkz(rad * cs, rad * sn);
}

int gaussian_fill(zd* X, int64_t ld, int64_t m, int64_t n, uint64_t seed, uint64_t offset,
                  cudaStream_t s) {
  const int64_t tot = m * n;
  if (tot <= 0) return 0;
  k_gauss<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(X, ld, m, n, seed, offset);
  note_launch();
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) { set_error(cudaGetErrorString(err)); return 3; }
  return 0;
}

__global__ void k_axpby(int64_t m, zd a, const zd* X, int64_t ldx, zd b, zd* Y, int64_t ldy) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t c = blockIdx.y;
  if (i >= m) return;
  zd y = mkz(0.0);
  if (b.x != 0.0 || b.y != 0.0) y = b * Y[c * ldy + i];
  Y[c * ldy + i] = y + a * X[c * ldx + i];
}

int axpby(int64_t m, int64_t n, zd a, const zd* X, int64_t ldx, zd b, zd* Y, int64_t ldy,
          cudaStream_t s) {
  for (int64_t c0 = 0; c0 < n; c0 += 65535) {
    int64_t cc = std::min<int64_t>(65535, n - c0);
    dim3 g((unsigned)((m + 255) / 256), (unsigned)cc);
    k_axpby<<<g, 256, 0, s>>>(m, a, X + c0 * ldx, ldx, b, Y + c0 * ldy, ldy);
    note_launch();
  }
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) { set_error(cudaGetErrorString(err)); return 3; }
  return 0;
}

// =========================================================================== Gram matrix X^H X
// Tall-skinny X (m x b, b <= 64): CTAs take row chunks and write partial
// b x b Grams, a second kernel sums the partials (fixed order: deterministic).
constexpr int GRAM_ROWS = 256;

// Partial Gram sums over GRAM_ROWS rows: only the upper triangle i <= j of the
// Hermitian b x b result is formed (pair index p -> column j = row of the
// triangular numbers, row i = p - j (j + 1) / 2); both halves are written.  A CTA
// takes GRAM_PAIRS pairs, two lanes each (real and imaginary part), so that the
// FP64 work of a row chunk (528 pairs at b = 32) spreads over nine CTAs instead of
// one: at N = 2777 eleven CTAs took 185 us a product, 38 so.  GRAM_STAGES tiles are in
// flight (cp.async): with plain loads between the tiles' barriers most of the time was
// the loads' latency.  Bound: the chain of 512 dependent FMA (17 us) for few rows, the FP64
// pipe for many, which needs warps on all four quarters of the SM and nothing on the pipe
// but the FMA.  32 pairs a CTA, four stages (one CTA of two warps a SM at b = 64) and the
// sign of the imaginary part as an FP64 negation took 2338 us at N = 32768, b = 64, where
// one CTA a chunk took 593; now 521 (435 is the pipe's time for it), 162 at b = 32.
constexpr int GRAM_PAIRS = 64, GRAM_TILE = 32, GRAM_STAGES = 2;
__global__ void __launch_bounds__(2 * GRAM_PAIRS) k_gram_partial(const zd* X, int64_t ld, int64_t m, int b, zd* part) {
  extern __shared__ zd gram_s[];   // [stage][column][GRAM_TILE + 1]
  const int64_t r0 = (int64_t)blockIdx.x * GRAM_ROWS, r1 = min(m, r0 + GRAM_ROWS);
  const int tid = threadIdx.x, im = tid & 1;
  const int npairs = b * (b + 1) / 2, p = blockIdx.y * GRAM_PAIRS + (tid >> 1);
  int j = (int)((sqrtf(8.f * (float)p + 1.f) - 1.f) * 0.5f);
  while (j * (j + 1) / 2 > p) --j;
  while ((j + 1) * (j + 2) / 2 <= p) ++j;
  const bool ok = p < npairs;
  const int i = ok ? p - j * (j + 1) / 2 : 0;
  if (!ok) j = 0;
  __shared__ int jmax;             // the columns past the CTA's last pair are not read
  if (tid == 0) jmax = 0;
  __syncthreads();
  if (ok) atomicMax(&jmax, j);
  __syncthreads();
  const int nc = jmax + 1;
  const int tiles = (int)((r1 - r0 + GRAM_TILE - 1) / GRAM_TILE);
  auto fetch = [&](int t) {
    if (t < tiles) {
      zd* dst = gram_s + (size_t)(t % GRAM_STAGES) * b * (GRAM_TILE + 1);
      for (int u = tid; u < GRAM_TILE * nc; u += blockDim.x) {
        const int c = u / GRAM_TILE, r = u % GRAM_TILE;
        const int64_t row = r0 + (int64_t)t * GRAM_TILE + r;
        const unsigned d = (unsigned)__cvta_generic_to_shared(dst + c * (GRAM_TILE + 1) + r);
        const zd* src = X + (int64_t)c * ld + (row < m ? row : 0);
        asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(row < m ? 16 : 0) : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");   // one group per tile, also past the last
  };
  for (int t = 0; t < GRAM_STAGES - 1; ++t) fetch(t);
  double acc = 0.0;
  const int sgn = im ? (int)0x80000000 : 0;
  for (int t = 0; t < tiles; ++t) {
    asm volatile("cp.async.wait_group %0;" ::"n"(GRAM_STAGES - 2) : "memory");
    __syncthreads();               // tile t is there; tile t - 1's stage is free
    fetch(t + GRAM_STAGES - 1);
    const zd* xi = gram_s + ((size_t)(t % GRAM_STAGES) * b + i) * (GRAM_TILE + 1);
    const zd* xj = gram_s + ((size_t)(t % GRAM_STAGES) * b + j) * (GRAM_TILE + 1);
    // conj(x_i) x_j with the operations of zfma: re: fma(x, u, fma(y, v, re)); im: fma(x, v, fma(-y, u, im)),
    // -y by its sign bit (a selected negation would run on the FP64 pipe)
#pragma unroll 8
    for (int r = 0; r < GRAM_TILE; ++r) {
      const zd a = xi[r], c = xj[r];
      const double y = __hiloint2double(__double2hiint(a.y) ^ sgn, __double2loint(a.y));
      acc = fma(a.x, im ? c.y : c.x, fma(y, im ? c.x : c.y, acc));
    }
  }
  const double other = __shfl_xor_sync(0xffffffffu, acc, 1);
  if (!ok || im) return;
  zd* P = part + (int64_t)blockIdx.x * b * b;
  P[j * b + i] = mkz(acc, other);
  if (i != j) P[i * b + j] = mkz(acc, -other);
}

__global__ void k_gram_reduce(const zd* part, int nparts, int b, zd* G) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= b * b) return;
  zd s = mkz(0.0);
#pragma unroll 8
  for (int p = 0; p < nparts; ++p) s += part[(int64_t)p * b * b + t];
  G[t] = s;
}

int gram_matrix(const zd* X, int64_t ld, int64_t m, int b, zd* G, zd* work, cudaStream_t s) {
  if (b > 64) { set_error("gram_matrix: b <= 64"); return 1; }
  const int nparts = (int)((m + GRAM_ROWS - 1) / GRAM_ROWS);
  static DeviceOnce attr;
  if (attr.need()) {
    cudaError_t e = cudaFuncSetAttribute(k_gram_partial, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(zd) * GRAM_STAGES * 64 * (GRAM_TILE + 1));
    if (e != cudaSuccess) { set_error(std::string("gram: ") + cudaGetErrorString(e)); return 3; }
    attr.done();
  }
  k_gram_partial<<<dim3((unsigned)nparts, (unsigned)((b * (b + 1) / 2 + GRAM_PAIRS - 1) / GRAM_PAIRS)), 2 * GRAM_PAIRS,
                   sizeof(zd) * GRAM_STAGES * b * (GRAM_TILE + 1), s>>>(X, ld, m, b, work);
  note_launch();
  k_gram_reduce<<<(b * b + 255) / 256, 256, 0, s>>>(work, nparts, b, G);
  note_launch();
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) { set_error(std::string("gram: ") + cudaGetErrorString(err)); return 3; }
  return 0;
}

// =========================================================================== pivoted Cholesky
// On a Hermitian b x b matrix (column-major, ld = b, b <= 64), one CTA, the
// matrix held in shared memory.  After return: rank r, perm[0:b], and R
// (upper, row j holds R[j, j..b-1] in permuted order) in Gm's upper triangle.
// Pivot: the largest remaining diagonal entry, the first of equal ones; the
// factorisation stops when it is <= rel_tol^2 times the first pivot (or <= 0).
// Bound: the chain of b steps (110 us at b = 32 with six barriers a step).  The pivot
// search compares bit patterns (non-negative doubles order like integers), warp 0 takes
// the pivot's root and reciprocal with it, the swap and the scaling of row j touch
// disjoint elements per thread and share a phase, and the Schur update packs the
// triangle's elements into full warps (an FP64 instruction costs its warp the same with
// one lane or 32).
__global__ void __launch_bounds__(512) k_pchol(zd* Gm, int b, double rel_tol, int* perm, int* rank_out) {
  extern __shared__ zd G[];
  __shared__ double dmax_s, rjj_s, rinv_s;
  __shared__ int piv_s, perm_s[64];
  const int tid = threadIdx.x;
  for (int u = tid; u < b * b; u += blockDim.x) G[u] = Gm[u];
  for (int i = tid; i < b; i += blockDim.x) perm_s[i] = i;
  __syncthreads();
  int rank = b;
  for (int j = 0; j < b; ++j) {
    if (tid < 32) {
      // warp argmax over the remaining diagonal; ties go to the lower index, NaN and
      // entries below zero are never taken
      long long v = -1;
      int p = INT_MAX;
      for (int i = j + tid; i < b; i += 32) {
        const long long d = __double_as_longlong(G[i * b + i].x);
        if (d > v && d <= 0x7ff0000000000000ll) { v = d; p = i; }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const long long v2 = __shfl_xor_sync(0xffffffffu, v, o);
        const int p2 = __shfl_xor_sync(0xffffffffu, p, o);
        if (v2 > v || (v2 == v && p2 < p)) { v = v2; p = p2; }
      }
      const double best = v < 0 ? -1.0 : __longlong_as_double(v);
      if (j == 0 && tid == 0) dmax_s = best;
      __syncwarp();
      const bool stop = best <= rel_tol * rel_tol * dmax_s || best <= 0.0;
      const double rjj = sqrt(best), rinv = 1.0 / rjj;
      if (tid == 0) {
        piv_s = stop ? -1 : p;
        rjj_s = rjj;
        rinv_s = rinv;
      }
    }
    __syncthreads();
    const int p = piv_s;
    if (p < 0) { rank = j; break; }
    // symmetric swap of rows and columns j and p, then row j of R:
    // R[j, i] = G[j, i] / rjj (G[j, i] at column i, row j), R[j, j] = rjj.  Thread i
    // touches G[j, i], G[p, i], G[i, j], G[i, p]; thread p the four corners.
    for (int i = tid; i < b; i += blockDim.x) {
      if (i == j) continue;
      zd rji = G[i * b + j];
      if (p != j) {
        if (i == p) {
          const zd cpj = G[j * b + p];
          G[p * b + p] = G[j * b + j];
          G[j * b + p] = rji;
          rji = cpj;
          const int t = perm_s[j];
          perm_s[j] = perm_s[p];
          perm_s[p] = t;
        } else {
          const zd t = G[j * b + i];
          G[j * b + i] = G[p * b + i];
          G[p * b + i] = t;
          const zd u = G[i * b + p];
          G[i * b + p] = rji;
          rji = u;
        }
      }
      G[i * b + j] = i > j ? rinv_s * rji : rji;
    }
    __syncthreads();
    if (tid == 0) G[j * b + j] = mkz(rjj_s);   // read by nobody before the next barrier
    // Schur complement: G[l, i] -= conj(R[j, l]) R[j, i] for j < l <= i, mirrored into
    // the lower triangle, which the pivot swaps read
    const int w = b - 1 - j;
    for (int u = tid; u < w * (w + 1) / 2; u += blockDim.x) {
      int di = (int)((sqrtf(8.f * (float)u + 1.f) - 1.f) * 0.5f);
      while (di * (di + 1) / 2 > u) --di;
      while ((di + 1) * (di + 2) / 2 <= u) ++di;
      const int i = j + 1 + di, l = j + 1 + u - di * (di + 1) / 2;
      const zd rji = G[i * b + j];
      const zd v = G[i * b + l] - conj(G[l * b + j]) * rji;
      G[i * b + l] = v;
      if (l < i) G[l * b + i] = conj(v);
    }
    __syncthreads();
  }
  __syncthreads();
  for (int u = tid; u < b * b; u += blockDim.x) Gm[u] = G[u];
  for (int i = tid; i < b; i += blockDim.x) perm[i] = perm_s[i];
  if (tid == 0) *rank_out = rank;
}

int pivoted_cholesky(zd* Gm, int b, double rel_tol, int* perm, int* rank_dev, cudaStream_t s) {
  if (b < 1 || b > 64) { set_error("pivoted_cholesky: 1 <= b <= 64"); return 1; }
  const int smem = (int)sizeof(zd) * b * b;
  static DeviceOnce attr;
  if (attr.need()) {
    cudaError_t e = cudaFuncSetAttribute(k_pchol, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(zd) * 64 * 64);
    if (e != cudaSuccess) { set_error(std::string("pivoted_cholesky: ") + cudaGetErrorString(e)); return 3; }
    attr.done();
  }
  k_pchol<<<1, 512, smem, s>>>(Gm, b, rel_tol, perm, rank_dev);
  note_launch();
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) { set_error(cudaGetErrorString(err)); return 3; }
  return 0;
}

// Y(i, 0:r) = X(i, perm[0:r]) R^{-1}, R the r x r upper factor of k_pchol
// (R[i][l] at R[l * b + i]).  Two kernels: Z = R^{-1} column by column (CTA c
// solves R z = e_c by back substitution, the update of each finished entry
// spread over the threads), then Y = X_perm Z over row tiles, where each row
// is independent: no dependency chain through memory, so the FP64 pipe is
// the bound.
__global__ void k_tri_inv(const zd* R, int b, const int* rank_dev, zd* Z) {
  extern __shared__ zd Rs[];   // R[0:c+1, 0:c+1], column-major, ld c + 1 (64 KB at c = 63)
  __shared__ zd dinv[64], zl_s;
  const int r = *rank_dev, c = blockIdx.x, i = threadIdx.x, n = c + 1;
  if (c >= r) return;
  for (int u = i; u < n * n; u += blockDim.x) {
    const int row = u % n, col = u / n;
    Rs[u] = (row <= col) ? R[col * b + row] : mkz(0.0);
  }
  if (i < n) dinv[i] = zrecip(R[i * b + i]);
  __syncthreads();
  zd s = mkz(i == c ? 1.0 : 0.0);
  for (int l = c; l >= 0; --l) {
    if (i == l) {
      zl_s = s * dinv[l];
      Z[c * r + l] = zl_s;
    }
    __syncthreads();
    const zd z = zl_s;
    if (i < l) s -= Rs[l * n + i] * z;
    __syncthreads();
  }
  for (int u = c + 1 + i; u < r; u += blockDim.x) Z[c * r + u] = mkz(0.0);
}

constexpr int TRSM_ROWS = 32;   // rows per CTA

// 4 warps: warp g forms columns g, g + 4, ..., g + 60 of 32 rows (interleaved,
// so the triangle's work is even over the warps), each column over its own
// l <= c only (a predicated-off FP64 FMA still takes its issue slot in the
// FP64 pipe); X tile and Z in shared memory (Z read as broadcasts, X
// row-consecutive across the lanes).
__global__ void __launch_bounds__(128) k_trsm_apply(const zd* X, int64_t ldx, int64_t m, const zd* Z,
                                                    const int* perm, const int* rank_dev, zd* Y,
                                                    int64_t ldy) {
  extern __shared__ zd sm[];
  const int r = *rank_dev;
  zd* Zs = sm;                 // r x r, column-major
  zd* xs = sm + r * r;         // r x TRSM_ROWS
  const int tid = threadIdx.x, lane = tid & 31, g = tid >> 5;
  const int64_t row0 = (int64_t)blockIdx.x * TRSM_ROWS;
  for (int u = tid; u < r * r; u += blockDim.x) Zs[u] = Z[u];
  for (int u = tid; u < r * TRSM_ROWS; u += blockDim.x) {
    const int l = u / TRSM_ROWS, rr = u % TRSM_ROWS;
    xs[u] = (row0 + rr < m) ? X[(int64_t)perm[l] * ldx + row0 + rr] : mkz(0.0);
  }
  __syncthreads();
  const int64_t i = row0 + lane;
  for (int c = g; c < r; c += 4) {
    // two partial sums (even and odd l) for two independent FMA chains
    zd a0 = mkz(0.0), a1 = mkz(0.0);
    const zd* zc = Zs + c * r;
    int l = 0;
    for (; l + 1 <= c; l += 2) {
      zfma(a0, xs[l * TRSM_ROWS + lane], zc[l]);
      zfma(a1, xs[(l + 1) * TRSM_ROWS + lane], zc[l + 1]);
    }
    if (l == c) zfma(a0, xs[l * TRSM_ROWS + lane], zc[l]);
    if (i < m) Y[(int64_t)c * ldy + i] = a0 + a1;
  }
}

int trsm_right_upper(const zd* X, int64_t ldx, int64_t m, const zd* R, int b, const int* perm,
                     const int* rank_dev, int rank_host, zd* Y, int64_t ldy, zd* work, cudaStream_t s) {
  if (b > 64 || rank_host > b) { set_error("trsm: block too wide"); return 1; }
  if (rank_host <= 0) return 0;
  static DeviceOnce attr;
  if (attr.need()) {
    cudaError_t e = cudaFuncSetAttribute(k_trsm_apply, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(sizeof(zd) * (64 * 64 + 64 * TRSM_ROWS)));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_tri_inv, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(sizeof(zd) * 64 * 64));
    if (e != cudaSuccess) { set_error(std::string("trsm: ") + cudaGetErrorString(e)); return 3; }
    attr.done();
  }
  k_tri_inv<<<(unsigned)rank_host, 64, sizeof(zd) * rank_host * rank_host, s>>>(R, b, rank_dev, work);
  note_launch();
  const size_t smem = sizeof(zd) * ((size_t)rank_host * rank_host + (size_t)rank_host * TRSM_ROWS);
  k_trsm_apply<<<(unsigned)((m + TRSM_ROWS - 1) / TRSM_ROWS), 128, smem, s>>>(X, ldx, m, work, perm, rank_dev,
                                                                                Y, ldy);
  note_launch();
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) { set_error(std::string("trsm: ") + cudaGetErrorString(err)); return 3; }
  return 0;
}

// =========================================================================== Gauss-Jordan inverse
// M = [A | I] (n x 2n, column-major, ld = n).  Step j: pick the pivot row in
// column j, swap, scale the pivot row, eliminate column j from every other row.
//
// One launch a step: CTA c owns a column right of j (the columns up to j are not read
// again, so column j itself stays as it is while all CTAs read it).  Each finds the pivot
// for itself, so no step waits for a kernel that runs on one SM: pivot and update kernels
// took 11 + 4 us a step at n = 90.
__global__ void __launch_bounds__(256) k_gj_step(zd* M, int64_t n, int64_t j, int* info, double* minpiv) {
  __shared__ long long key_s[8];
  __shared__ int idx_s[8];
  __shared__ zd inv_s;
  const int tid = threadIdx.x;
  const zd* cj = M + j * n;
  zd* col = M + (j + 1 + blockIdx.x) * n;
  // largest |entry|^2 of column j from row j on, the first of equal ones; squares compare
  // like their bit patterns, NaN is never taken
  long long key = -1;
  int p = INT_MAX;
  for (int64_t i = j + tid; i < n; i += blockDim.x) {
    const long long v = __double_as_longlong(abs2(cj[i]));
    if (v > key && v <= 0x7ff0000000000000ll) { key = v; p = (int)i; }
  }
  auto take = [&](long long k2, int p2) {
    if (k2 > key || (k2 == key && p2 < p)) { key = k2; p = p2; }
  };
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    take(__shfl_xor_sync(0xffffffffu, key, o), __shfl_xor_sync(0xffffffffu, p, o));
  if ((tid & 31) == 0) { key_s[tid >> 5] = key; idx_s[tid >> 5] = p; }
  __syncthreads();
  for (int w = 0; w < 8; ++w) take(key_s[w], idx_s[w]);
  if (key < 0) p = (int)j;
  if (tid == 0) {
    inv_s = key > 0 ? zrecip(cj[p]) : mkz(0.0);
    if (blockIdx.x == 0) {
      const double pv = sqrt(key < 0 ? -1.0 : __longlong_as_double(key));
      if (pv < *minpiv) *minpiv = pv;
      if (!(pv > 0.0)) *info = (int)j + 1;
    }
  }
  const zd mj = col[j], mp = col[p];
  __syncthreads();   // row j and the pivot's row of this column are read
  const zd rowj = mp * inv_s;
  for (int64_t i = tid; i < n; i += blockDim.x) {
    if (i == j) { col[i] = rowj; continue; }
    zd v = i == p ? mj : col[i];
    v -= (i == p ? cj[j] : cj[i]) * rowj;
    col[i] = v;
  }
}

__global__ void k_identity(zd* M, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) M[i * n + i] = mkz(1.0);
}

int lu_inverse(zd* A, int64_t n, zd* Ainv, zd* work, int* info_dev, double* minpiv_dev, cudaStream_t s) {
  zd* M = work;
  cudaMemcpy2DAsync(M, sizeof(zd) * n, A, sizeof(zd) * n, sizeof(zd) * n, n, cudaMemcpyDeviceToDevice, s);
  cudaMemsetAsync(M + n * n, 0, sizeof(zd) * n * n, s);
  k_identity<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(M + n * n, n);
  note_launch();
  const double big = 1e300;
  cudaMemcpyAsync(minpiv_dev, &big, sizeof(double), cudaMemcpyHostToDevice, s);
  cudaMemsetAsync(info_dev, 0, sizeof(int), s);
  for (int64_t j = 0; j < n; ++j) {
    k_gj_step<<<(unsigned)(2 * n - 1 - j), 256, 0, s>>>(M, n, j, info_dev, minpiv_dev);
    note_launch();
  }
  cudaMemcpy2DAsync(Ainv, sizeof(zd) * n, M + n * n, sizeof(zd) * n, sizeof(zd) * n, n,
                    cudaMemcpyDeviceToDevice, s);
  cudaError_t err = cudaStreamSynchronize(s);
  if (err != cudaSuccess) { set_error(std::string("inverse: ") + cudaGetErrorString(err)); return 3; }
  return 0;
}

}  // namespace wcs
