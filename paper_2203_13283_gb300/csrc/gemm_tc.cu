// Tensor-core contraction for the mixed-precision form: the sampling of the
// skeleton (Eq. 7), the preconditioned right-hand side of Eq. (5) and the
// operator applies of Eq. (6) are dense complex products with the assembled
// Galerkin matrices, carried out here as real products on the 5th-generation
// tensor cores of sm_103a.
//
//   D (M x Nc, FP32) = sum_p  A_{ia[p]} (M x K) * B_{ib[p]} (Nc x K)^T
//
// A and B are bf16 "planes" (split-bf16: x = hi + lo [+ lo2]), K-major (row
// major with K contiguous).  Tiles of A (128 x 64) and B (NT x 64) are staged
// by TMA (128-byte swizzle) into a multi-stage shared-memory ring guarded by
// mbarriers; one thread issues tcgen05.mma (kind::f16, M = 128, N = NT,
// K = 16) accumulating in TMEM; tcgen05.commit releases ring slots; the four
// warps drain TMEM with tcgen05.ld in the epilogue, which applies a complex
// combination (see Epi) and writes FP32 or FP64 output.
//
// Every wait on an mbarrier is bounded; on expiry the kernel records an error
// code in *err, stops issuing work, waits (bounded) for its own copies and
// MMAs, frees TMEM and returns, so the host sees WCS_ERR_TIMEOUT.
#include <cuda.h>

#include <algorithm>

#include "gemm_tc.h"
#include "tc_ptx.cuh"

namespace wcs {

// ----------------------------------------------------------------------------- kernel
constexpr int TC_THREADS = 128;

template <int NT, int PA, int PB, int STAGES>
struct TcSmem {
  static constexpr int A_BYTES = TC_BM * TC_BK * 2;   // 16 KB
  static constexpr int B_BYTES = NT * TC_BK * 2;      // 16 or 32 KB
  static constexpr int STAGE_BYTES = PA * A_BYTES + PB * B_BYTES;
  static constexpr int TOTAL = STAGES * STAGE_BYTES + 1024 /*align*/ + 256 /*barriers, flags*/;
};

template <int NT, int PA, int PB, int STAGES>
__global__ void __launch_bounds__(TC_THREADS, 1)
    k_gemm_tc(const __grid_constant__ CUtensorMap mA0, const __grid_constant__ CUtensorMap mA1,
              const __grid_constant__ CUtensorMap mA2, const __grid_constant__ CUtensorMap mB0,
              const __grid_constant__ CUtensorMap mB1, const __grid_constant__ CUtensorMap mB2, TcArgs args) {
  using L = TcSmem<NT, PA, PB, STAGES>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + STAGES * L::STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* done = empty + STAGES;
  uint32_t* tslot = (uint32_t*)(done + 1);
  volatile int* abort_flag = (volatile int*)(tslot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.y * TC_BM;
  const int n0 = blockIdx.x * NT;
  // split-K: CTA z takes k-blocks [z kper, (z + 1) kper); the host picks kper
  // so that every split is non-empty
  const int nk_all = (args.K + TC_BK - 1) / TC_BK;
  const int kb0 = (args.kper > 0) ? (int)blockIdx.z * args.kper : 0;
  const int nk = (args.kper > 0) ? min(args.kper, nk_all - kb0) : nk_all;

  if (tc_given_up(args.err)) return;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    mbar_init(done, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"((uint32_t)NT));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;

  const CUtensorMap* mapA[3] = {&mA0, &mA1, &mA2};
  const CUtensorMap* mapB[3] = {&mB0, &mB1, &mB2};
  // instruction descriptor: D f32, A bf16, B bf16, both K-major, N, M
  const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(NT >> 3) << 17) |
                         ((uint32_t)(TC_BM >> 4) << 24);

  volatile int* issued = (volatile int*)(tslot + 2);     // k-blocks whose loads were issued
  volatile int* consumed = (volatile int*)(tslot + 3);   // k-blocks the MMA thread waited for
  if (threadIdx.x == 0) { *issued = 0; *consumed = 0; }
  __syncthreads();
  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer
    for (int kb = 0; kb < nk; ++kb) {
      const int s = kb % STAGES;
      if (kb >= STAGES) {
        if (!mbar_wait(&empty[s], ((kb / STAGES) + 1) & 1, WAIT_LIMIT, args.err)) { *abort_flag = 11; break; }
      }
      if (*abort_flag) break;
      uint8_t* st = smem + s * L::STAGE_BYTES;
      mbar_expect_tx(&full[s], L::STAGE_BYTES);
      const int k0 = (kb0 + kb) * TC_BK;
#pragma unroll
      for (int p = 0; p < PA; ++p) tma_load_2d(st + p * L::A_BYTES, mapA[p], &full[s], k0, m0);
#pragma unroll
      for (int p = 0; p < PB; ++p) tma_load_2d(st + PA * L::A_BYTES + p * L::B_BYTES, mapB[p], &full[s], k0, n0);
      *issued = kb + 1;
    }
  } else if (warp == 1 && lane == 0) {
    // ---------------- MMA issuer
    for (int kb = 0; kb < nk; ++kb) {
      const int s = kb % STAGES;
      if (!mbar_wait(&full[s], (kb / STAGES) & 1, WAIT_LIMIT, args.err)) { *abort_flag = 12; break; }
      *consumed = kb + 1;
      if (*abort_flag) break;
      tc_fence_after();
      uint8_t* st = smem + s * L::STAGE_BYTES;
      for (int p = 0; p < args.nprod; ++p) {
        const uint8_t* ta = st + args.ia[p] * L::A_BYTES;
        const uint8_t* tb = st + PA * L::A_BYTES + args.ib[p] * L::B_BYTES;
        const uint64_t da = sw128_desc(ta), db = sw128_desc(tb);
#pragma unroll
        for (int kk = 0; kk < TC_BK / 16; ++kk) {
          // advance 16 bf16 = 32 bytes along K inside the swizzle atom
          mma_bf16(tmem, da + (uint64_t)(2 * kk), db + (uint64_t)(2 * kk), idesc,
                   (kb > 0 || p > 0 || kk > 0) ? 1u : 0u);
        }
      }
      mma_commit(&empty[s]);
    }
    mma_commit(done);   // arrives once every MMA issued above has completed
  }
  __syncwarp();
  // ---------------- epilogue: all four warps
  bool got = mbar_wait(done, 0, WAIT_LIMIT, args.err);
  const bool waited = __all_sync(0xffffffffu, got);
  got = waited && (__shfl_sync(0xffffffffu, *abort_flag, 0) == 0);
  tc_fence_after();
  if (!got) {
    if (!waited && lane == 0) atomicCAS((int*)abort_flag, 0, 13);
    __syncwarp();
    if (threadIdx.x == 0) {
      const int zero_flag = 0;
      atomicExch(args.err, 1000 * (*abort_flag) + (int)(blockIdx.x % 1000));
      // let the loads already in flight land before the CTA's shared memory goes away
      for (int kb = *consumed; kb < *issued; ++kb)
        (void)mbar_wait(&full[kb % STAGES], (kb / STAGES) & 1, WAIT_LIMIT, &zero_flag);
    }
  } else {
    const int row = m0 + warp * 32 + lane;   // TMEM lane = tile row
#pragma unroll 1
    for (int c0 = 0; c0 < NT; c0 += 32) {
      float v[32];
      tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, v);
      if (args.ws) {
        // split-K partial, column-major [split][Nc][M]: a warp writes 32 consecutive rows per column
        if (row < args.M) {
          float* w = args.ws + (int64_t)blockIdx.z * args.Nc * args.M + row;
#pragma unroll
          for (int i = 0; i < 32; ++i)
            if (n0 + c0 + i < args.Nc) w[(int64_t)(n0 + c0 + i) * args.M] = v[i];
        }
      } else {
        epilogue_store(args, row, n0 + c0, v);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)NT));
  }
}

// ----------------------------------------------------------------------------- host side
template <int NT, int PA, int PB, int STAGES>
static int launch_tc(const TcOperand& A, const TcOperand& B, TcArgs& args, cudaStream_t s) {
  using L = TcSmem<NT, PA, PB, STAGES>;
  CUtensorMap ma[3], mb[3];
  std::memset(ma, 0, sizeof(ma));
  std::memset(mb, 0, sizeof(mb));
  for (int p = 0; p < PA; ++p) TRY_TC(make_map(&ma[p], A.plane[p], args.M, args.K, A.ld, TC_BM));
  for (int p = 0; p < PB; ++p) TRY_TC(make_map(&mb[p], B.plane[p], args.Nc, args.K, B.ld, NT));
  for (int p = PA; p < 3; ++p) ma[p] = ma[0];
  for (int p = PB; p < 3; ++p) mb[p] = mb[0];
  auto kern = k_gemm_tc<NT, PA, PB, STAGES>;
  static DeviceOnce attr;   // one instance per template instantiation
  if (attr.need()) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, L::TOTAL);
    if (e != cudaSuccess) { set_error(std::string("gemm_tc: shared-memory opt-in: ") + cudaGetErrorString(e)); return 3; }
    attr.done();
  }
  const int nk = (args.K + TC_BK - 1) / TC_BK;
  const int splits = (args.kper > 0) ? (nk + args.kper - 1) / args.kper : 1;
  dim3 grid((unsigned)((args.Nc + NT - 1) / NT), (unsigned)((args.M + TC_BM - 1) / TC_BM), (unsigned)splits);
  kern<<<grid, TC_THREADS, L::TOTAL, s>>>(ma[0], ma[1], ma[2], mb[0], mb[1], mb[2], args);
  note_launch();
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { set_error(std::string("gemm_tc launch: ") + cudaGetErrorString(e)); return 3; }
  return 0;
}

// A sum of FP32 values as FP32 terms (Knuth's error-free TwoSum).  Converting and adding
// every value on the FP64 pipe took 50 us for the partials of 4096 x 256 and seven splits.
// Three terms lose no value's last bit: FP64's sum or better, for the one-accumulator
// products, whose partials FP64 summed.  Two terms (~48 bits) for the drained products,
// whose parts of K were FP32 register sums before they were split; the third would cost
// 1.2% of a solve of 360 columns at N = 4096.
template <bool THREE>
struct FloatSum {
  float a = 0.f, b = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float s = a + x, u = s - a, e = (a - (s - u)) + (x - u);
    a = s;
    const float t = b + e;
    if (THREE) {
      const float v = t - b;
      c += (b - (t - v)) + (e - v);
    }
    b = t;
  }
  // infinities, NaN and sums beyond the FP32 range are left to an FP64 sum
  __device__ __forceinline__ bool ok() const { return fabsf(a) <= 3.402823466e38f; }
  __device__ __forceinline__ double value() const {
    return epi_f32_to_f64(a) + (THREE ? epi_f32_to_f64(b) + epi_f32_to_f64(c) : epi_f32_to_f64(b));
  }
};

// Sum of the split-K partials in a fixed order and the epilogue.
template <bool DRAINED>
__global__ void k_splitk_reduce(TcArgs a, int splits) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t plane = (int64_t)a.Nc * a.M;
  if (a.epi == EPI_RAW_F64) {
    if (t >= plane) return;
    const int row = (int)(t % a.M), col = (int)(t / a.M);
    double sum = 0.0;
#pragma unroll 8
    for (int z = 0; z < splits; ++z) sum += (double)a.ws[z * plane + t];
    double* o = (double*)a.out + (int64_t)row * a.ldo + col;
    *o = a.alpha.x * sum + ((a.beta.x == 0.0) ? 0.0 : a.beta.x * (*o));
    return;
  }
  const int ncols = a.Nc / 2;
  if (t >= (int64_t)a.M * ncols) return;
  const int row = (int)(t % a.M), j = (int)(t / a.M);
  const float* w = a.ws + (int64_t)(2 * j) * a.M + row;
  FloatSum<!DRAINED> r, s;
#pragma unroll 8
  for (int z = 0; z < splits; ++z) {
    r.add(w[z * plane]);
    s.add(w[z * plane + a.M]);
  }
  double re = r.value(), im = s.value();
  if (!r.ok() || !s.ok()) {
    re = im = 0.0;
    for (int z = 0; z < splits; ++z) {
      re += (double)w[z * plane];
      im += (double)w[z * plane + a.M];
    }
  }
  if (a.conj_out) im = -im;
  zd* o = (zd*)a.out + (int64_t)j * a.ldo + row;
  if (epi_unit(a)) {   // as epilogue_store: an infinite part must not meet the zero of alpha
    zd p = a.alpha.x < 0.0 ? mkz(-re, -im) : mkz(re, im);
    if (a.beta.x == 1.0) {
      const zd q = *o;
      p.x += q.x;
      p.y += q.y;
    }
    *o = p;
    return;
  }
  zd p = a.alpha * mkz(re, im);
  if (!(a.beta.x == 0.0 && a.beta.y == 0.0)) p += a.beta * (*o);
  *o = p;
}


// ----------------------------------------------------------------------------- accurate variant
// The tensor-core accumulator truncates: its relative error grows with the
// number of accumulation steps (measured ~3e-8 per step).  This variant keeps
// each K = 16 step's result in its own TMEM buffer (two buffers, ping-pong),
// and eight drain warps move it into FP32 registers before the next use, so no
// TMEM sum spans more than one step.  Register sums are two-level (an inner
// sum over 64 steps folded into an outer sum), which keeps the FP32 rounding
// of ~K/16 additions near 1e-7 at a quarter of the cost of compensated
// summation.  Tile 128 x 128; warps 0-7 drain (warp w: TMEM lanes 32 (w % 4),
// columns 64 (w / 4)), warp 8 loads (TMA), warp 9 issues the MMAs.  The drain
// is bound by the latency of the TMEM load, so each warp moves its 64 columns
// in one load and keeps only the inner sums in registers; the outer sums live
// in the last 128 TMEM columns, after three step buffers (384 columns).
constexpr int ACC_NT = 128, ACC_THREADS = 320, ACC_FOLD = 64, ACC_NBUF = 3;
constexpr int ACC_OUTER = ACC_NBUF * ACC_NT;   // first TMEM column of the outer sums

template <int PA, int PB, int STAGES>
struct AccSmem {
  static constexpr int A_BYTES = TC_BM * TC_BK * 2;        // 16 KB
  static constexpr int B_BYTES = ACC_NT * TC_BK * 2;       // 16 KB
  static constexpr int STAGE_BYTES = PA * A_BYTES + PB * B_BYTES;
  static constexpr int TOTAL = STAGES * STAGE_BYTES + 1024 + 256;
};

// K splits of a launch (the host picks kper so that every split has work)
static unsigned tc_splits(const TcArgs& a) {
  const int nk = (a.K + TC_BK - 1) / TC_BK;
  return a.kper > 0 ? (unsigned)((nk + a.kper - 1) / a.kper) : 1u;
}

// 32 columns of one row: the epilogue, or the split's FP32 partial, column-major
// [split][Nc][M] (a warp writes 32 consecutive rows per column)
__device__ __forceinline__ void tile_store(const TcArgs& a, int row, int col0, const float (&v)[32]) {
  if (!a.ws) {
    epilogue_store(a, row, col0, v);
    return;
  }
  if (row >= a.M) return;
  float* w = a.ws + (int64_t)blockIdx.z * a.Nc * a.M + row;
#pragma unroll
  for (int i = 0; i < 32; ++i)
    if (col0 + i < a.Nc) w[(int64_t)(col0 + i) * a.M] = v[i];
}

template <int PA, int PB, int STAGES>
__global__ void __launch_bounds__(ACC_THREADS, 1)
    k_gemm_tc_acc(const __grid_constant__ CUtensorMap mA0, const __grid_constant__ CUtensorMap mA1,
                  const __grid_constant__ CUtensorMap mA2, const __grid_constant__ CUtensorMap mB0,
                  const __grid_constant__ CUtensorMap mB1, const __grid_constant__ CUtensorMap mB2, TcArgs args) {
  using L = AccSmem<PA, PB, STAGES>;
  extern __shared__ uint8_t smem_raw[];
  if (tc_given_up(args.err)) return;
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + STAGES * L::STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* tfull = empty + STAGES;      // [ACC_NBUF] MMA -> drain
  uint64_t* tempty = tfull + ACC_NBUF;   // [ACC_NBUF] drain -> MMA
  uint32_t* tslot = (uint32_t*)(tempty + ACC_NBUF);
  volatile int* abort_flag = (volatile int*)(tslot + 1);
  volatile int* issued = (volatile int*)(tslot + 2);
  volatile int* consumed = (volatile int*)(tslot + 3);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.y * TC_BM;
  const int n0 = blockIdx.x * ACC_NT;
  const int nk_all = (args.K + TC_BK - 1) / TC_BK;
  const int kb0 = (args.kper > 0) ? (int)blockIdx.z * args.kper : 0;   // split-K: k-blocks [kb0, kb0 + nk)
  const int nk = (args.kper > 0) ? min(args.kper, nk_all - kb0) : nk_all;
  const int nsteps = nk * (TC_BK / 16);
  // accumulation groups: `drain` consecutive K = 16 steps share one TMEM
  // buffer before it is drained (1: every step)
  const int drain = args.drain > 1 ? args.drain : 1;
  const int ngroups = (nsteps + drain - 1) / drain;

  if (threadIdx.x == 0) {
    for (int q = 0; q < STAGES; ++q) { mbar_init(&full[q], 1); mbar_init(&empty[q], 1); }
    for (int q = 0; q < ACC_NBUF; ++q) { mbar_init(&tfull[q], 1); mbar_init(&tempty[q], 8); }
    *abort_flag = 0;
    *issued = 0;
    *consumed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(512u));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;
  const CUtensorMap* mapA[3] = {&mA0, &mA1, &mA2};
  const CUtensorMap* mapB[3] = {&mB0, &mB1, &mB2};
  const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(ACC_NT >> 3) << 17) |
                         ((uint32_t)(TC_BM >> 4) << 24);

  float inner[64];
#pragma unroll
  for (int i = 0; i < 64; ++i) inner[i] = 0.f;

  if (warp == 8) {
    if (lane == 0) {
      for (int kb = 0; kb < nk; ++kb) {
        const int st = kb % STAGES;
        if (kb >= STAGES) {
          if (!mbar_wait(&empty[st], ((kb / STAGES) + 1) & 1, WAIT_LIMIT, args.err)) { *abort_flag = 21; break; }
        }
        if (*abort_flag) break;
        uint8_t* sp = smem + st * L::STAGE_BYTES;
        mbar_expect_tx(&full[st], L::STAGE_BYTES);
        const int k0 = (kb0 + kb) * TC_BK;
#pragma unroll
        for (int p = 0; p < PA; ++p) tma_load_2d(sp + p * L::A_BYTES, mapA[p], &full[st], k0, m0);
#pragma unroll
        for (int p = 0; p < PB; ++p) tma_load_2d(sp + PA * L::A_BYTES + p * L::B_BYTES, mapB[p], &full[st], k0, n0);
        *issued = kb + 1;
      }
    }
  } else if (warp == 9) {
    if (lane == 0) {
      // products of order < planes, smallest first (the order of tc_products,
      // checked on the host); descriptors are formed once per stage and the
      // group/buffer counters advance without divisions, so the issuing thread
      // keeps ahead of the tensor core
      constexpr int NP = (PA == 3) ? 6 : 3;
      constexpr int IA[6] = {PA == 3 ? 2 : 1, PA == 3 ? 1 : 0, 0, 1, 0, 0};
      constexpr int IB[6] = {0, 1, PA == 3 ? 2 : 0, 0, 1, 0};
      int b = 0, ingroup = 0, q = 0;
      bool ok = true;
      for (int kb = 0; kb < nk && ok; ++kb) {
        const int st = kb % STAGES;
        if (!mbar_wait(&full[st], (kb / STAGES) & 1, WAIT_LIMIT, args.err)) { *abort_flag = 22; break; }
        *consumed = kb + 1;
        if (*abort_flag) break;
        tc_fence_after();
        const uint8_t* sp = smem + st * L::STAGE_BYTES;
        uint64_t da[NP], db[NP];
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          da[p] = sw128_desc(sp + IA[p] * L::A_BYTES);
          db[p] = sw128_desc(sp + PA * L::A_BYTES + IB[p] * L::B_BYTES);
        }
        if (drain == TC_BK / 16) {
          // one group per stage, issued product-major: every step's small
          // plane products enter the fresh accumulator before any large one,
          // so the truncating accumulator cuts them at their own scale, not
          // at the scale of the leading product
          if (q >= ACC_NBUF) {
            if (!mbar_wait(&tempty[b], ((q / ACC_NBUF) - 1) & 1, WAIT_LIMIT, args.err)) {
              *abort_flag = 25;
              mma_commit(&empty[st]);
              break;
            }
            tc_fence_after();
          }
          const uint32_t dt = tmem + (uint32_t)(b * ACC_NT);
#pragma unroll
          for (int p = 0; p < NP; ++p)
#pragma unroll
            for (int kk = 0; kk < TC_BK / 16; ++kk)
              mma_bf16(dt, da[p] + (uint64_t)(2 * kk), db[p] + (uint64_t)(2 * kk), idesc,
                       (p == 0 && kk == 0) ? 0u : 1u);
          mma_commit(&tfull[b]);
          ++q;
          b = (b == ACC_NBUF - 1) ? 0 : b + 1;
          mma_commit(&empty[st]);
          continue;
        }
#pragma unroll
        for (int kk = 0; kk < TC_BK / 16; ++kk) {
          if (ingroup == 0 && q >= ACC_NBUF) {
            if (!mbar_wait(&tempty[b], ((q / ACC_NBUF) - 1) & 1, WAIT_LIMIT, args.err)) {
              *abort_flag = 25; ok = false; break;
            }
            tc_fence_after();
          }
          const uint32_t dt = tmem + (uint32_t)(b * ACC_NT);
#pragma unroll
          for (int p = 0; p < NP; ++p)
            mma_bf16(dt, da[p] + (uint64_t)(2 * kk), db[p] + (uint64_t)(2 * kk), idesc,
                     (ingroup == 0 && p == 0) ? 0u : 1u);
          ++ingroup;
          if (ingroup == drain || (kb == nk - 1 && kk == TC_BK / 16 - 1)) {
            mma_commit(&tfull[b]);
            ingroup = 0;
            ++q;
            b = (b == ACC_NBUF - 1) ? 0 : b + 1;
          }
        }
        mma_commit(&empty[st]);
      }
    }
  } else {
    // drain warps
    const int lanebase = 32 * (warp & 3), colhalf = 64 * (warp >> 2);
    const uint32_t touter = tmem + ((uint32_t)lanebase << 16) + (uint32_t)(ACC_OUTER + colhalf);
    float v[64];
#pragma unroll
    for (int i = 0; i < 64; ++i) v[i] = 0.f;
    tmem_st64(touter, v);
    for (int g = 0; g < ngroups; ++g) {
      const int b = g % ACC_NBUF;
      bool got = (drain > 1) ? mbar_wait_sleep(&tfull[b], (g / ACC_NBUF) & 1, WAIT_LIMIT, args.err, 256u)
                             : mbar_wait(&tfull[b], (g / ACC_NBUF) & 1, WAIT_LIMIT, args.err);
      got = __all_sync(0xffffffffu, got) && (__shfl_sync(0xffffffffu, *abort_flag, 0) == 0);
      if (!got) { if (lane == 0) atomicCAS((int*)abort_flag, 0, 24); break; }
      tc_fence_after();
      tmem_ld64(tmem + ((uint32_t)lanebase << 16) + (uint32_t)(b * ACC_NT + colhalf), v);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&tempty[b])) : "memory");
#pragma unroll
      for (int i = 0; i < 64; ++i) inner[i] += v[i];
      if ((g % ACC_FOLD) == ACC_FOLD - 1) {
        tmem_ld64(touter, v);
#pragma unroll
        for (int i = 0; i < 64; ++i) { v[i] += inner[i]; inner[i] = 0.f; }
        tmem_st64(touter, v);
      }
    }
  }
  __syncthreads();
  const bool ok = (*abort_flag == 0);
  if (!ok) {
    if (threadIdx.x == 0) {
      const int zero_flag = 0;
      atomicExch(args.err, 1000 * (*abort_flag) + (int)(blockIdx.x % 1000));
      for (int kb = *consumed; kb < *issued; ++kb)
        (void)mbar_wait(&full[kb % STAGES], (kb / STAGES) & 1, WAIT_LIMIT, &zero_flag);
    }
  } else if (warp < 8) {
    const int lanebase = 32 * (warp & 3), colhalf = 64 * (warp >> 2);
    float v[64], out[32];
    tmem_ld64(tmem + ((uint32_t)lanebase << 16) + (uint32_t)(ACC_OUTER + colhalf), v);
#pragma unroll
    for (int i = 0; i < 32; ++i) out[i] = v[i] + inner[i];
    tile_store(args, m0 + lanebase + lane, n0 + colhalf, out);
#pragma unroll
    for (int i = 0; i < 32; ++i) out[i] = v[32 + i] + inner[32 + i];
    tile_store(args, m0 + lanebase + lane, n0 + colhalf + 32, out);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u));
  }
}

template <int PA, int PB, int STAGES>
static int launch_tc_acc(const TcOperand& A, const TcOperand& B, TcArgs& args, cudaStream_t s) {
  using L = AccSmem<PA, PB, STAGES>;
  CUtensorMap ma[3], mb[3];
  std::memset(ma, 0, sizeof(ma));
  std::memset(mb, 0, sizeof(mb));
  for (int p = 0; p < PA; ++p) TRY_TC(make_map(&ma[p], A.plane[p], args.M, args.K, A.ld, TC_BM));
  for (int p = 0; p < PB; ++p) TRY_TC(make_map(&mb[p], B.plane[p], args.Nc, args.K, B.ld, ACC_NT));
  for (int p = PA; p < 3; ++p) ma[p] = ma[0];
  for (int p = PB; p < 3; ++p) mb[p] = mb[0];
  auto kern = k_gemm_tc_acc<PA, PB, STAGES>;
  static DeviceOnce attr;   // one instance per template instantiation
  if (attr.need()) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, L::TOTAL);
    if (e != cudaSuccess) { set_error(std::string("gemm_tc: shared-memory opt-in: ") + cudaGetErrorString(e)); return 3; }
    attr.done();
  }
  dim3 grid((unsigned)((args.Nc + ACC_NT - 1) / ACC_NT), (unsigned)((args.M + TC_BM - 1) / TC_BM), tc_splits(args));
  kern<<<grid, ACC_THREADS, L::TOTAL, s>>>(ma[0], ma[1], ma[2], mb[0], mb[1], mb[2], args);
  note_launch();
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { set_error(std::string("gemm_tc_acc launch: ") + cudaGetErrorString(e)); return 3; }
  return 0;
}

// ----------------------------------------------------------------------------- periodic drain, wide tile
// The periodic mode (two planes, three products, accumulator drained every
// `drain` K = 16 steps) on 128 x 256 tiles.  With 128 x 128 tiles its three
// products per 64 KB stage (96 flop per staged byte) starved the tensor pipe
// on the L2-to-shared-memory feed; 128 x 256 tiles carry 131 flop per byte,
// like the one-accumulator kernel.  Two TMEM accumulators of 256 columns fill
// the 512 TMEM columns, so the drained sums stay in registers: warp w of the
// eight drain warps owns TMEM lanes 32 (w % 4) and columns 128 (w / 4), 128
// FP32 sums per thread.  A single level of sums suffices: K / (16 drain)
// additions (64 at K = 65536) round far below this mode's ~1e-5.
constexpr int PER_NT = 256, PER_THREADS = 320;

template <int STAGES>
struct PerSmem {
  static constexpr int A_BYTES = TC_BM * TC_BK * 2;        // 16 KB
  static constexpr int B_BYTES = PER_NT * TC_BK * 2;       // 32 KB
  static constexpr int STAGE_BYTES = 2 * A_BYTES + 2 * B_BYTES;
  static constexpr int TOTAL = STAGES * STAGE_BYTES + 1024 + 256;
};

template <int STAGES>
__global__ void __launch_bounds__(PER_THREADS, 1)
    k_gemm_tc_per(const __grid_constant__ CUtensorMap mA0, const __grid_constant__ CUtensorMap mA1,
                  const __grid_constant__ CUtensorMap mB0, const __grid_constant__ CUtensorMap mB1, TcArgs args) {
  using L = PerSmem<STAGES>;
  extern __shared__ uint8_t smem_raw[];
  if (tc_given_up(args.err)) return;
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + STAGES * L::STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* tfull = empty + STAGES;      // [2] MMA -> drain
  uint64_t* tempty = tfull + 2;          // [2] drain -> MMA
  uint32_t* tslot = (uint32_t*)(tempty + 2);
  volatile int* abort_flag = (volatile int*)(tslot + 1);
  volatile int* issued = (volatile int*)(tslot + 2);
  volatile int* consumed = (volatile int*)(tslot + 3);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.y * TC_BM;
  const int n0 = blockIdx.x * PER_NT;
  const int nk_all = (args.K + TC_BK - 1) / TC_BK;
  const int kb0 = (args.kper > 0) ? (int)blockIdx.z * args.kper : 0;
  const int nk = (args.kper > 0) ? min(args.kper, nk_all - kb0) : nk_all;
  const int nsteps = nk * (TC_BK / 16);
  const int drain = args.drain > 1 ? args.drain : 1;
  const int ngroups = (nsteps + drain - 1) / drain;

  if (threadIdx.x == 0) {
    for (int q = 0; q < STAGES; ++q) { mbar_init(&full[q], 1); mbar_init(&empty[q], 1); }
    for (int q = 0; q < 2; ++q) { mbar_init(&tfull[q], 1); mbar_init(&tempty[q], 8); }
    *abort_flag = 0;
    *issued = 0;
    *consumed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(512u));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;
  const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(PER_NT >> 3) << 17) |
                         ((uint32_t)(TC_BM >> 4) << 24);

  float sum[128];
#pragma unroll
  for (int i = 0; i < 128; ++i) sum[i] = 0.f;

  if (warp == 8) {
    if (lane == 0) {
      for (int kb = 0; kb < nk; ++kb) {
        const int st = kb % STAGES;
        if (kb >= STAGES) {
          if (!mbar_wait(&empty[st], ((kb / STAGES) + 1) & 1, WAIT_LIMIT, args.err)) { *abort_flag = 31; break; }
        }
        if (*abort_flag) break;
        uint8_t* sp = smem + st * L::STAGE_BYTES;
        mbar_expect_tx(&full[st], L::STAGE_BYTES);
        const int k0 = (kb0 + kb) * TC_BK;
        tma_load_2d(sp, &mA0, &full[st], k0, m0);
        tma_load_2d(sp + L::A_BYTES, &mA1, &full[st], k0, m0);
        tma_load_2d(sp + 2 * L::A_BYTES, &mB0, &full[st], k0, n0);
        tma_load_2d(sp + 2 * L::A_BYTES + L::B_BYTES, &mB1, &full[st], k0, n0);
        *issued = kb + 1;
      }
    }
  } else if (warp == 9) {
    if (lane == 0) {
      // products of order < 2, smallest first: A1 B0, A0 B1, A0 B0
      constexpr int IA[3] = {1, 0, 0};
      constexpr int IB[3] = {0, 1, 0};
      int b = 0, ingroup = 0, q = 0;
      bool ok = true;
      for (int kb = 0; kb < nk && ok; ++kb) {
        const int st = kb % STAGES;
        if (!mbar_wait(&full[st], (kb / STAGES) & 1, WAIT_LIMIT, args.err)) { *abort_flag = 32; break; }
        *consumed = kb + 1;
        if (*abort_flag) break;
        tc_fence_after();
        const uint8_t* sp = smem + st * L::STAGE_BYTES;
        uint64_t da[3], db[3];
#pragma unroll
        for (int p = 0; p < 3; ++p) {
          da[p] = sw128_desc(sp + IA[p] * L::A_BYTES);
          db[p] = sw128_desc(sp + 2 * L::A_BYTES + IB[p] * L::B_BYTES);
        }
#pragma unroll
        for (int kk = 0; kk < TC_BK / 16; ++kk) {
          if (ingroup == 0 && q >= 2) {
            if (!mbar_wait(&tempty[b], ((q / 2) - 1) & 1, WAIT_LIMIT, args.err)) {
              *abort_flag = 35; ok = false; break;
            }
            tc_fence_after();
          }
          const uint32_t dt = tmem + (uint32_t)(b * PER_NT);
#pragma unroll
          for (int p = 0; p < 3; ++p)
            mma_bf16(dt, da[p] + (uint64_t)(2 * kk), db[p] + (uint64_t)(2 * kk), idesc,
                     (ingroup == 0 && p == 0) ? 0u : 1u);
          ++ingroup;
          if (ingroup == drain || (kb == nk - 1 && kk == TC_BK / 16 - 1)) {
            mma_commit(&tfull[b]);
            ingroup = 0;
            ++q;
            b ^= 1;
          }
        }
        mma_commit(&empty[st]);
      }
    }
  } else {
    // drain warps: sums of their 32 lanes x 128 columns in registers
    const int lanebase = 32 * (warp & 3), colbase = 128 * (warp >> 2);
    for (int g = 0; g < ngroups; ++g) {
      const int b = g & 1;
      bool got = mbar_wait_sleep(&tfull[b], (g >> 1) & 1, WAIT_LIMIT, args.err, 256u);
      got = __all_sync(0xffffffffu, got) && (__shfl_sync(0xffffffffu, *abort_flag, 0) == 0);
      if (!got) { if (lane == 0) atomicCAS((int*)abort_flag, 0, 34); break; }
      tc_fence_after();
#pragma unroll
      for (int c4 = 0; c4 < 4; ++c4) {
        float v[32];
        tmem_ld32(tmem + ((uint32_t)lanebase << 16) + (uint32_t)(b * PER_NT + colbase + 32 * c4), v);
#pragma unroll
        for (int i = 0; i < 32; ++i) sum[32 * c4 + i] += v[i];
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&tempty[b])) : "memory");
    }
  }
  __syncthreads();
  const bool ok = (*abort_flag == 0);
  if (!ok) {
    if (threadIdx.x == 0) {
      const int zero_flag = 0;
      atomicExch(args.err, 1000 * (*abort_flag) + (int)(blockIdx.x % 1000));
      for (int kb = *consumed; kb < *issued; ++kb)
        (void)mbar_wait(&full[kb % STAGES], (kb / STAGES) & 1, WAIT_LIMIT, &zero_flag);
    }
  } else if (warp < 8) {
    const int lanebase = 32 * (warp & 3), colbase = 128 * (warp >> 2);
#pragma unroll
    for (int c4 = 0; c4 < 4; ++c4) {
      float out[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) out[i] = sum[32 * c4 + i];
      tile_store(args, m0 + lanebase + lane, n0 + colbase + 32 * c4, out);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u));
  }
}

template <int STAGES>
static int launch_tc_per(const TcOperand& A, const TcOperand& B, TcArgs& args, cudaStream_t s) {
  using L = PerSmem<STAGES>;
  CUtensorMap ma[2], mb[2];
  std::memset(ma, 0, sizeof(ma));
  std::memset(mb, 0, sizeof(mb));
  for (int p = 0; p < 2; ++p) TRY_TC(make_map(&ma[p], A.plane[p], args.M, args.K, A.ld, TC_BM));
  for (int p = 0; p < 2; ++p) TRY_TC(make_map(&mb[p], B.plane[p], args.Nc, args.K, B.ld, PER_NT));
  auto kern = k_gemm_tc_per<STAGES>;
  static DeviceOnce attr;
  if (attr.need()) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, L::TOTAL);
    if (e != cudaSuccess) { set_error(std::string("gemm_tc: shared-memory opt-in: ") + cudaGetErrorString(e)); return 3; }
    attr.done();
  }
  dim3 grid((unsigned)((args.Nc + PER_NT - 1) / PER_NT), (unsigned)((args.M + TC_BM - 1) / TC_BM), tc_splits(args));
  kern<<<grid, PER_THREADS, L::TOTAL, s>>>(ma[0], ma[1], mb[0], mb[1], args);
  note_launch();
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { set_error(std::string("gemm_tc_per launch: ") + cudaGetErrorString(e)); return 3; }
  return 0;
}

static int launch_splitk_reduce(const TcArgs& args, int splits, bool drained, cudaStream_t s) {
  const int64_t n = (int64_t)args.M * ((args.epi == EPI_RAW_F64) ? args.Nc : args.Nc / 2);
  const unsigned blocks = (unsigned)((n + 255) / 256);
  if (drained) k_splitk_reduce<true><<<blocks, 256, 0, s>>>(args, splits);
  else k_splitk_reduce<false><<<blocks, 256, 0, s>>>(args, splits);
  note_launch();
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { set_error(std::string("split-K reduce: ") + cudaGetErrorString(e)); return 3; }
  return 0;
}

// k-blocks per split of a drained product (0: no split).  A launch takes whole
// waves of 152 CTAs, so a grid of 24 or 192 tiles leaves most of the chip idle in
// its only or last wave; splitting K evens it out at the price of the partials
// (written and read once, FP32) and of a prologue and epilogue per
// CTA.  Microseconds: a K = 64 block of a 128 x 128 tile is 0.8 with three planes
// (24 MMAs of 64 clocks) and 0.4 with two, of a 128 x 256 tile with two 0.8; about
// 4 per CTA; 8 bytes per partial at 5 TB/s and a 4 us reduction launch.
static int acc_kper(const TcArgs& a, int nt, int planes) {
  if (!a.ws || !(a.epi == EPI_RAW_F64 || (a.epi == EPI_CPLX_F64 && (a.Nc % 2) == 0))) return 0;
  const int nk = (a.K + TC_BK - 1) / TC_BK;
  const int64_t tiles = (int64_t)((a.Nc + nt - 1) / nt) * ((a.M + TC_BM - 1) / TC_BM);
  const double block = (planes == 3 || nt == PER_NT) ? 0.8 : 0.4, part = 8.0e-6 / 5.0 * (double)a.M * a.Nc;
  double best = 1e300;
  int kper = 0;
  for (int sp = 1; sp <= std::min(64, nk / 4 > 0 ? nk / 4 : 1); ++sp) {
    if (sp > 1 && (int64_t)sp * a.Nc * a.M > a.ws_elems) break;
    const int per = (nk + sp - 1) / sp;
    const double t = (double)((tiles * sp + 151) / 152) * (per * block + 4.0) + (sp > 1 ? sp * part + 4.0 : 0.0);
    if (t < best) { best = t; kper = sp > 1 ? per : 0; }
  }
  return kper;
}

int gemm_tc_accurate(const TcOperand& A, const TcOperand& B, TcArgs args, cudaStream_t s) {
  if (args.M <= 0 || args.Nc <= 0 || args.K <= 0) return 0;
  if (args.nprod < 1 || args.nprod > 6) { set_error("gemm_tc: 1..6 products"); return 1; }
  for (int p = 0; p < args.nprod; ++p)
    if (args.ia[p] >= A.planes || args.ib[p] >= B.planes) { set_error("gemm_tc: plane index"); return 1; }
  if ((args.M + TC_BM - 1) / TC_BM > 65535) { set_error("gemm_tc: M too large"); return 1; }
  {
    // the kernel issues the full product list of tc_products for its plane count
    TcArgs ref;
    tc_products(A.planes, ref);
    bool same = (A.planes == B.planes) && (args.nprod == ref.nprod);
    for (int p = 0; same && p < ref.nprod; ++p) same = (args.ia[p] == ref.ia[p] && args.ib[p] == ref.ib[p]);
    if (!same) { set_error("gemm_tc_accurate: needs the full product list of tc_products"); return 1; }
  }
  // two planes drained every 16 or more steps on a grid of more than one
  // column tile: the wide-tile kernel
  const bool wide = A.planes == 2 && B.planes == 2 && args.drain >= 16 && args.Nc > 128;
  args.kper = acc_kper(args, wide ? PER_NT : ACC_NT, A.planes);
  if (args.kper == 0) args.ws = nullptr;
  const int splits = (int)tc_splits(args);
  int r = 1;
  if (A.planes == 3 && B.planes == 3) r = launch_tc_acc<3, 3, 2>(A, B, args, s);
  else if (wide) r = launch_tc_per<2>(A, B, args, s);
  else if (A.planes == 2 && B.planes == 2) r = launch_tc_acc<2, 2, 3>(A, B, args, s);
  else set_error("gemm_tc_accurate: plane combination not built");
  if (r || splits == 1) return r;
  return launch_splitk_reduce(args, splits, true, s);
}

int gemm_tc_split_plan(int M, int Nc, int K, int planesA, int planesB, int epi, int64_t* ws_elems) {
  *ws_elems = 0;
  if (M <= 0 || Nc <= 0 || K <= 0) return 0;
  if (!(epi == EPI_RAW_F64 || (epi == EPI_CPLX_F64 && (Nc % 2) == 0))) return 0;
  const int NT = ((planesA == 3 && planesB == 3) || Nc <= 128) ? 128 : 256;
  const int nk = (K + TC_BK - 1) / TC_BK;
  const int64_t ctas = (int64_t)((Nc + NT - 1) / NT) * ((M + TC_BM - 1) / TC_BM);
  if (ctas >= 152 || nk < 8) return 0;
  int64_t want = (2 * 152 + ctas - 1) / ctas;
  want = std::min<int64_t>(want, nk / 4);
  // at most 64 MB of partials
  want = std::min<int64_t>(want, ((int64_t)1 << 24) / ((int64_t)Nc * M));
  if (want <= 1) return 0;
  const int kper = (int)((nk + want - 1) / want);
  const int splits = (nk + kper - 1) / kper;   // <= want, every split non-empty
  *ws_elems = (int64_t)splits * Nc * M;
  return kper;
}

int gemm_tc(const TcOperand& A, const TcOperand& B, TcArgs args, cudaStream_t s) {
  if (args.M <= 0 || args.Nc <= 0 || args.K <= 0) return 0;
  if (args.nprod < 1 || args.nprod > 6) { set_error("gemm_tc: 1..6 products"); return 1; }
  if (A.planes < 1 || A.planes > 3 || B.planes < 1 || B.planes > 3) { set_error("gemm_tc: 1..3 planes"); return 1; }
  for (int p = 0; p < args.nprod; ++p)
    if (args.ia[p] >= A.planes || args.ib[p] >= B.planes) { set_error("gemm_tc: plane index"); return 1; }
  if ((args.M + TC_BM - 1) / TC_BM > 65535) { set_error("gemm_tc: M too large"); return 1; }
  const int key = A.planes * 10 + B.planes;
  const int NT = (key == 33 || args.Nc <= 128) ? 128 : 256;
  // split-K when the output tiles cannot fill the GPU (tall-K products such
  // as Q^H Y with few rows); needs the caller's FP32 workspace
  float* ws = args.ws;
  args.ws = nullptr;
  args.kper = 0;
  int splits = 1;
  if (ws && args.force_kper > 0) {
    const int nk = (args.K + TC_BK - 1) / TC_BK;
    const int kper = args.force_kper;
    splits = (nk + kper - 1) / kper;
    if ((int64_t)splits * args.Nc * args.M > args.ws_elems) { set_error("gemm_tc: split-K workspace too small"); return 1; }
    args.kper = kper;
    args.ws = ws;
  } else if (ws) {
    int64_t need = 0;
    const int kper = gemm_tc_split_plan(args.M, args.Nc, args.K, A.planes, B.planes, args.epi, &need);
    if (kper > 0 && need <= args.ws_elems) {
      args.kper = kper;
      args.ws = ws;
      const int nk = (args.K + TC_BK - 1) / TC_BK;
      splits = (nk + kper - 1) / kper;
    }
  }
  int r = 0;
  switch (key) {
    case 11: r = (NT == 128) ? launch_tc<128, 1, 1, 4>(A, B, args, s) : launch_tc<256, 1, 1, 4>(A, B, args, s); break;
    case 22: r = (NT == 128) ? launch_tc<128, 2, 2, 3>(A, B, args, s) : launch_tc<256, 2, 2, 2>(A, B, args, s); break;
    case 33: r = launch_tc<128, 3, 3, 2>(A, B, args, s); break;
    default: set_error("gemm_tc: plane combination not built"); return 1;
  }
  if (r || args.no_reduce || splits == 1) return r;
  return launch_splitk_reduce(args, splits, false, s);
}

}  // namespace wcs
