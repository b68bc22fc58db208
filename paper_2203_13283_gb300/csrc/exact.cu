// Exact real contraction on the tensor cores (wcs_gemm_exact); the solver's own exact
// products run in fxgemm.cu.
//
// A split-bf16 product accumulated in FP32 carries ~1e-7 relative error.  This file
// evaluates a product without rounding error on the same tensor cores:
//
//  * every row of an operand is cut into chunks of EX_CHUNK consecutive K
//    elements; each chunk gets a power-of-two scale 2^E (its largest entry
//    below 2^E), and the scaled entries, all in (-1, 1), are written as
//    EX_SLICES fixed-point slices of 7 bits, y = sum_s y_s 2^-7(s+1) with
//    integers |y_0| <= 128 and |y_s| <= 64, each exact in bf16;
//  * a product of two slices is a sum of integer products (<= 2^14 each);
//    over one chunk of 1024 terms it stays below 2^24, where the tensor core's
//    FP32 accumulation is exact, so the contraction runs split-K with one
//    split per chunk and returns exact integer partial sums;
//  * the partials are scaled by 2^(E_A + E_B) and summed over the chunks in
//    float-float (an exact integer below 2^24 times a power of two is exact
//    in FP32, and TwoSum keeps ~48 bits of the running sum on the FP32 pipe,
//    which runs at 64 times the FP64 rate of this GPU); each pair's sum, times
//    2^-7(s+t+2), is added to the FP64 output.
//
// Pairs with s + t < EX_LEVELS are formed (21 of the 36); the dropped ones are
// below 2^-56 of the chunk scales.
#include <cuda_bf16.h>

#include "gemm_tc.h"
#include "exact.h"

namespace wcs {

__device__ __forceinline__ uint16_t int_bf16(double v) {
  return __bfloat16_as_ushort(__double2bfloat16(v));   // exact for integers |v| <= 256
}

constexpr int EX_PER = EX_CHUNK / 256;   // values per thread of a 256-thread block

// 2^e as a float for the normal range (e in [-126, 127]); scaled partials of
// the residual products stay far inside it (operator entries and currents
// between ~1e-12 and ~1e3, partial sums below 2^24)
__device__ __forceinline__ float pow2f(int e) {
  e = max(-126, min(127, e));
  return __int_as_float((e + 127) << 23);
}

// (hi, lo) += v with TwoSum (Knuth): hi + lo carries the sum to ~2^-48
__device__ __forceinline__ void ff_acc(float2& a, float v) {
  const float s = a.x + v;
  const float bb = s - a.x;
  const float err = (a.x - (s - bb)) + (v - bb);
  a.x = s;
  a.y += err;
}

// Exponent E of a chunk held by the block (EX_PER values per thread):
// max |v| < 2^E, or 0 for an all-zero chunk.  Written to *expo by thread 0.
__device__ __forceinline__ int chunk_exponent(const double (&m)[EX_PER], int16_t* expo) {
  __shared__ double red[8];
  __shared__ int eshared;
  double x = 0.0;
#pragma unroll
  for (int t = 0; t < EX_PER; ++t) x = fmax(x, m[t]);
  for (int o = 16; o > 0; o >>= 1) x = fmax(x, __shfl_xor_sync(0xffffffffu, x, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
  __syncthreads();
  if (threadIdx.x == 0) {
    double mm = 0.0;
    for (int w = 0; w < 8; ++w) mm = fmax(mm, red[w]);
    eshared = (mm > 0.0) ? ilogb(mm) + 1 : 0;   // mm < 2^E
    *expo = (int16_t)eshared;
  }
  __syncthreads();
  return eshared;
}

// The EX_SLICES fixed-point slices of v / 2^E at offset `off` of each slice plane.
__device__ __forceinline__ void write_slices(double v, int E, uint16_t* const* slice, int64_t off) {
  double r = ldexp(v, 7 - E);   // in (-128, 128); exact scaling
#pragma unroll
  for (int q = 0; q < EX_SLICES; ++q) {
    const double y = rint(r);
    slice[q][off] = int_bf16(y);
    r = (r - y) * 128.0;          // exact: r - y in [-1/2, 1/2], 7 more bits
  }
}

// Real FP64 rows (row-major, ld): one block per (row, chunk).
__global__ void __launch_bounds__(256) k_slice_real(const double* X, int64_t K, int64_t ld, ExactOperand out) {
  const int64_t row = blockIdx.y, c = blockIdx.x;
  double v[EX_PER], m[EX_PER];
#pragma unroll
  for (int t = 0; t < EX_PER; ++t) {
    const int64_t k = c * EX_CHUNK + t * 256 + threadIdx.x;
    v[t] = (k < K) ? X[row * ld + k] : 0.0;
    m[t] = fabs(v[t]);
  }
  const int E = chunk_exponent(m, out.expo + row * out.nchunks + c);
#pragma unroll
  for (int t = 0; t < EX_PER; ++t) {
    const int64_t k = c * EX_CHUNK + t * 256 + threadIdx.x;
    if (k < out.ld) write_slices(v[t], E, out.slice, row * out.ld + k);
  }
}

// D (M x Nc, row-major ldd) op= weight * sum_c 2^(EA(i,c) + EB(j,c)) P[c][j][i].
__global__ void k_exact_reduce_real(const float* __restrict__ P, int splits, int M, int Nc, const int16_t* EA,
                                    const int16_t* EB, int64_t nchunks, double weight, int first, double* D,
                                    int64_t ldd) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)M * Nc) return;
  const int i = (int)(t % M), j = (int)(t / M);
  const int64_t plane = (int64_t)Nc * M;
  float2 sum = make_float2(0.f, 0.f);
  for (int c = 0; c < splits; ++c) {
    const float sc = pow2f((int)EA[(int64_t)i * nchunks + c] + (int)EB[(int64_t)j * nchunks + c]);
    ff_acc(sum, P[c * plane + (int64_t)j * M + i] * sc);
  }
  const double acc = (double)sum.x + (double)sum.y;
  double* o = D + (int64_t)i * ldd + j;
  *o = first ? weight * acc : *o + weight * acc;
}

int exact_operand_alloc_bytes(int64_t rows, int64_t K, int64_t* ld, int64_t* nchunks, size_t* slice_bytes,
                              size_t* expo_bytes) {
  *ld = ((K + 63) / 64) * 64;
  *nchunks = (K + EX_CHUNK - 1) / EX_CHUNK;
  *slice_bytes = sizeof(uint16_t) * (size_t)rows * (size_t)(*ld);
  *expo_bytes = sizeof(int16_t) * (size_t)rows * (size_t)(*nchunks);
  return 0;
}

int exact_slice_real(const double* X, int64_t rows, int64_t K, int64_t ld, const ExactOperand& out, cudaStream_t s) {
  for (int64_t r0 = 0; r0 < rows; r0 += 65535) {
    const int64_t rr = std::min<int64_t>(65535, rows - r0);
    ExactOperand o = out;
    for (int q = 0; q < EX_SLICES; ++q) o.slice[q] = out.slice[q] + r0 * out.ld;
    o.expo = out.expo + r0 * out.nchunks;
    dim3 g((unsigned)out.nchunks, (unsigned)rr);
    k_slice_real<<<g, 256, 0, s>>>(X + r0 * ld, K, ld, o);
    note_launch();
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { set_error(std::string("exact slices: ") + cudaGetErrorString(e)); return 3; }
  return 0;
}

int exact_product_real(const ExactOperand& A, int M, const ExactOperand& B, int Nc, int K, double* D, int64_t ldd,
                       float* ws, int64_t ws_elems, int* err, cudaStream_t s) {
  if (M <= 0 || Nc <= 0) return 0;
  bool first = true;
  for (int lev = EX_LEVELS - 1; lev >= 0; --lev) {
    for (int sa = 0; sa <= lev; ++sa) {
      const int sb = lev - sa;
      if (sa >= EX_SLICES || sb >= EX_SLICES) continue;
      TcOperand oa, ob;
      oa.planes = ob.planes = 1;
      oa.ld = A.ld;
      ob.ld = B.ld;
      oa.plane[0] = A.slice[sa];
      ob.plane[0] = B.slice[sb];
      TcArgs t;
      t.M = M;
      t.Nc = Nc;
      t.K = K;
      tc_products(1, t);
      t.epi = EPI_RAW_F64;
      t.err = err;
      t.ws = ws;
      t.ws_elems = ws_elems;
      t.force_kper = EX_CHUNK / 64;
      t.no_reduce = 1;
      TRY_TC(gemm_tc(oa, ob, t, s));
      const int64_t n = (int64_t)M * Nc;
      k_exact_reduce_real<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(ws, (int)A.nchunks, M, Nc, A.expo, B.expo,
                                                                      A.nchunks, ldexp(1.0, -7 * (lev + 2)),
                                                                      first ? 1 : 0, D, ldd);
      note_launch();
      first = false;
    }
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { set_error(std::string("exact product: ") + cudaGetErrorString(e)); return 3; }
  return 0;
}

}  // namespace wcs
