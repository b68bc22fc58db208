// Complex FP64 products (the operator products of Eq. (6) in the FP64 form, the
// projections of the skeleton of Eq. (7), the Woodbury products of Eq. (9), the
// far-field map) on the tensor cores.
//
// GB300 has 64 times fewer FP64 than FP32 lanes (1.25 TFLOP/s), but its tensor
// cores sum integer products exactly: a bf16 product of integers |a|, |b| <= 128
// is exact and the FP32 accumulator holds sums up to 2^24.  So each row of an
// operand is scaled by a power of two (its largest entry below 2^E) and written
// as NS signed 8-bit digits, v = sum_s d_s 2^(E - 6 - 8 s), |d_s| <= 128.
//
//             digits NS  error of v    levels s + t  digit pairs  dropped pairs
//   products      8      2^(E - 63)       0 .. 7         36        7 2^-62
//   operators     6      2^(E - 47)       0 .. 6         26        4 2^-54   (times 2^(EA + EB) per term)
//
// Every level has its own TMEM accumulator, exact over FX_CHUNK stages (K = 128, where
// eight pairs of 128 products of 2^14 just reach 2^24).  Then it is drained: levels 0 .. 4
// into 64-bit integers, exact over any K, the three (six digits: two) levels below them
// into FP32 sums; rounded to FP64 once per split of K.
//
// The error of an entry is thus relative to the largest entries a of its row of A and b of
// its column of B.  Eight digits: k a b 2^-55 from the digits, whatever the order of the
// sum, and at most k a b 2^-55 (k / 64) from the FP32 sums, a bound that takes all lower
// digits coherent and every rounding one way; with digits as they come it is their roundings
// of ~sqrt(k) 2^-62 a b.  Six digits: k a b 2^-43.  The error of an FP64 dot product is up
// to 2 k 2^-53 sum_k |A_ik| |B_kj|.  For entries of similar size the digits' is the smaller
// one; entries below 2^-10 of their row's or column's largest keep fewer than 53
// bits, so where the large entries of a column meet small ones of the row (a column that
// spans many orders of magnitude), an FP64 product is the more accurate one.
//
// The complex product runs as the real product of A (m x 2k, re and im
// interleaved) with B' (2n x 2k; row 2j = (Re x, -Im x), row 2j + 1 =
// (Im x, Re x)).  Operands lie in memory as [row][K / 32][slice][32] bf16: one
// 128-byte row of a TMA box is two slices of 32 K-values, so a stage is
// NS / 2 boxes per operand and the swizzle atom is that of the other
// tensor-core kernels, the second slice 64 bytes into it.
//
// Tile 128 x 64: the levels, 64 columns each, fill 512 TMEM columns (seven with six
// digits: 448).  The MMAs of a stage run from the highest level down; each level is
// committed by itself, so the eight drain warps empty it while the next levels run.
// Warp 8 loads, warp 9 issues.  K is split over the grid (FP64 partials, summed in
// order) when the tiles alone do not fill the GPU.
//
// Bound: with eight digits 72 MMAs of 128 x 64 x 16 per 32 K-values (52 with six),
// limited by the shared-memory reads of A (6 KB per MMA, 48 clocks); for few columns
// the slicing of A, which reads 16 and writes 32 bytes per complex entry.
#include <algorithm>

#include "fxgemm.h"
#include "tc_ptx.cuh"

namespace wcs {

constexpr int FX_BM = 128, FX_BN = 64, FX_BK = 32, FX_CHUNK = 4, FX_THREADS = 320;
constexpr int FX_BAD = 1 << 20;                       // row exponent of a row that is not finite
template <int NS>
struct Fx {
  static constexpr int TOP = 8 * (NS - 1) + 6;        // fixed-point position: |v| 2^(TOP - E) < 2^TOP
  static constexpr int ROW = NS * FX_BK;              // bf16 values of one row and stage
  // digit-pair levels formed.  Six digits take one level past their own: without it the
  // dropped pairs, five of 2^-46 of the row scales a term, left an exact-residual solve at N = 16384
  // at 1.4e-11 where the entries' own 2^-48 leave 6e-13
  static constexpr int LEVELS = NS == 8 ? 8 : NS + 1;
  static constexpr int A_BYTES = FX_BM * ROW * 2, B_BYTES = FX_BN * ROW * 2;
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int STAGES = NS == 8 ? 2 : 3;
  static constexpr int SMEM = STAGES * STAGE_BYTES + 1024 + 512;
  static_assert(NS % 2 == 0 && LEVELS * FX_BN <= 512, "two slices per TMA row, one TMEM accumulator per level");
  static_assert((int64_t)NS * FX_CHUNK * FX_BK * (1 << 14) <= (1 << 24), "level sums stay exact in FP32");
};

// ----------------------------------------------------------------------------- slices
// Operand view: row i, complex K index t at p[i * si + t * sk].  dup: the B'
// operand (two real rows per view row).
struct FxSrc {
  const zd* p;
  int64_t si, sk;
  int conj, dup;
  int64_t rows, K, kb;   // complex K values, K / 32 stages of the real view
  uint16_t* d;           // [real row][kb][FX_SLICES][32]
  int* e;                // exponent per view row
  int kfast, segs;       // sk == 1; blocks that share a row (or a row group)
  int64_t blocks;
};

// The digits of v in a row of exponent E (|v| < 2^E), by integer operations on
// its bits (the FP64 pipe would take ~20 operations per value): rounded to the
// last digit, balanced digits -128..127 from the low end.
template <int NS>
__device__ __forceinline__ void fx_digits(double v, int E, int (&d)[NS]) {
  const long long u = __double_as_longlong(v);
  const int be = (int)((u >> 52) & 0x7FF);
  long long x = 0;
  if (be > 0) {
    const long long mant = (u & 0xFFFFFFFFFFFFFll) | (1ll << 52);
    const int sh = be - 1075 + Fx<NS>::TOP - E;    // v 2^(TOP - E) = mant 2^sh
    if (sh >= 0) x = mant << sh;              // below 2^TOP by the choice of E
    else if (sh >= -54) x = (mant + (1ll << (-sh - 1))) >> -sh;
    if (u < 0) x = -x;
  }
#pragma unroll
  for (int s = NS - 1; s > 0; --s) {
    d[s] = (int)(signed char)(x & 255);
    x = (x - d[s]) >> 8;
  }
  d[0] = (int)x;
}

// bf16 bits of an integer |d| <= 128 in the upper half of the word (exact)
__device__ __forceinline__ uint32_t fx_bf16_hi(int d) {
  return __float_as_uint(__int_as_float(0x4B400000 + d) - 12582912.f);
}
__device__ __forceinline__ uint32_t fx_pack(int a, int b) {
  return (fx_bf16_hi(a) >> 16) | (fx_bf16_hi(b) & 0xFFFF0000u);
}

__device__ __forceinline__ unsigned fx_mag(zd v) {
  return max((unsigned)__double2hiint(v.x) & 0x7FFFFFFFu, (unsigned)__double2hiint(v.y) & 0x7FFFFFFFu);
}
// exponent E with |v| < 2^E from the largest high word; zero and denormal rows: 0
__device__ __forceinline__ int fx_exp(unsigned hi) {
  const int be = (int)(hi >> 20);
  return be == 0x7FF ? FX_BAD : (be == 0 ? 0 : be - 1022);
}

template <int NS>
__device__ __forceinline__ void fx_write(const FxSrc& S, int64_t row, int64_t t, zd v, int E) {
  int re[NS], im[NS];
  if (E == FX_BAD) v = mkz(0.0);
  if (S.conj) v.y = -v.y;
  fx_digits<NS>(v.x, E, re);
  fx_digits<NS>(v.y, E, im);
  const int64_t in = (t >> 4) * Fx<NS>::ROW + 2 * (t & 15);
  if (!S.dup) {
    uint16_t* o = S.d + row * S.kb * Fx<NS>::ROW + in;
#pragma unroll
    for (int s = 0; s < NS; ++s) *(uint32_t*)(o + s * FX_BK) = fx_pack(re[s], im[s]);
  } else {
    uint16_t* o = S.d + 2 * row * S.kb * Fx<NS>::ROW + in;
    uint16_t* o1 = o + S.kb * Fx<NS>::ROW;
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      *(uint32_t*)(o + s * FX_BK) = fx_pack(re[s], -im[s]);
      *(uint32_t*)(o1 + s * FX_BK) = fx_pack(im[s], re[s]);
    }
  }
}

// Both operands of a product in one launch: blocks [0, a.blocks) slice a, the
// rest b.  A block reads its row(s) once for the largest magnitude and again
// (from L1 or L2) for the digits of its segment of K.
template <int NS>
__global__ void __launch_bounds__(256) k_fx_slice(FxSrc a, FxSrc b) {
  const bool first = (int64_t)blockIdx.x < a.blocks;
  const FxSrc& S = first ? a : b;
  const int64_t blk = first ? blockIdx.x : blockIdx.x - a.blocks;
  const int tid = threadIdx.x;
  const int64_t group = blk / S.segs;
  const int seg = (int)(blk - group * S.segs);
  const int64_t slots = S.kb * 16;                                      // complex K values with the padding
  const int64_t per = ((slots + S.segs - 1) / S.segs + 15) & ~(int64_t)15;
  const int64_t t0 = min(slots, seg * per), t1 = min(slots, t0 + per);
  __shared__ unsigned red[16];
  if (S.kfast) {
    // one row, K over the threads
    const zd* p = S.p + group * S.si;
    unsigned m = 0;
    for (int64_t t = tid; t < S.K; t += 256) m = max(m, fx_mag(p[t]));
    m = __reduce_max_sync(0xffffffffu, m);
    if ((tid & 31) == 0) red[tid >> 5] = m;
    __syncthreads();
    m = red[0];
#pragma unroll
    for (int w = 1; w < 8; ++w) m = max(m, red[w]);
    const int E = fx_exp(m);
    if (tid == 0 && seg == 0) S.e[group] = E;
    for (int64_t t = t0 + tid; t < t1; t += 256) fx_write<NS>(S, group, t, t < S.K ? p[t] : mkz(0.0), E);
  } else {
    // 16 rows, contiguous (or strided) across the low thread index; tiles of 16 x 16 turned in shared memory
    __shared__ zd tile[16][17];
    if (tid < 16) red[tid] = 0u;
    __syncthreads();
    const int r = tid & 15, kk = tid >> 4;
    const int64_t row = group * 16 + r;
    unsigned m = 0;
    if (row < S.rows)
      for (int64_t t = kk; t < S.K; t += 16) m = max(m, fx_mag(S.p[row * S.si + t * S.sk]));
    atomicMax(&red[r], m);
    __syncthreads();
    if (tid < 16 && seg == 0 && group * 16 + tid < S.rows) S.e[group * 16 + tid] = fx_exp(red[tid]);
    const int64_t wrow = group * 16 + kk;       // this thread writes row kk, K value r of each tile
    const int E = fx_exp(red[kk]);
    for (int64_t t = t0; t < t1; t += 16) {
      __syncthreads();
      tile[r][kk] = (row < S.rows && t + kk < S.K) ? S.p[row * S.si + (t + kk) * S.sk] : mkz(0.0);
      __syncthreads();
      if (wrow < S.rows) fx_write<NS>(S, wrow, t + r, tile[kk][r], E);
    }
  }
}

// Rows of an operand held as split-bf16 planes (row-major, ld values, K of them
// valid): value = sum of its planes.  One block per row; the leading plane alone
// fixes the exponent (the rest is below half a unit of its last place).
template <int NS>
__global__ void __launch_bounds__(256) k_fx_slice_planes(const uint16_t* p0, const uint16_t* p1, const uint16_t* p2,
                                                         int64_t K, int64_t ld, int64_t kb, uint16_t* d, int* e) {
  __shared__ unsigned red[8];
  const int64_t row = blockIdx.x;
  const int tid = threadIdx.x;
  const uint32_t* a0 = (const uint32_t*)(p0 + row * ld);
  const uint32_t* a1 = p1 ? (const uint32_t*)(p1 + row * ld) : nullptr;
  const uint32_t* a2 = p2 ? (const uint32_t*)(p2 + row * ld) : nullptr;
  const int64_t K2 = (K + 1) / 2;
  unsigned m = 0;
  for (int64_t t = tid; t < K2; t += 256) {
    const uint32_t w = a0[t];
    m = max(m, max(w & 0x7FFFu, (w >> 16) & 0x7FFFu));
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if ((tid & 31) == 0) red[tid >> 5] = m;
  __syncthreads();
  m = red[0];
#pragma unroll
  for (int w = 1; w < 8; ++w) m = max(m, red[w]);
  const int be = (int)(m >> 7);
  const int E = be == 255 ? FX_BAD : (be == 0 ? 0 : be - 126);   // |x| < 2^(be - 126)
  if (tid == 0) e[row] = E;
  uint16_t* o = d + row * kb * Fx<NS>::ROW;
  for (int64_t t = tid; t < kb * 16; t += 256) {
    const uint32_t w0 = t < K2 ? a0[t] : 0u, w1 = (a1 && t < K2) ? a1[t] : 0u, w2 = (a2 && t < K2) ? a2[t] : 0u;
    int u[NS], v[NS];
    double x = 0.0, y = 0.0;
    if (E != FX_BAD) {
      x = (double)__uint_as_float(w0 << 16) + (double)__uint_as_float(w1 << 16) + (double)__uint_as_float(w2 << 16);
      y = (double)__uint_as_float(w0 & 0xFFFF0000u) + (double)__uint_as_float(w1 & 0xFFFF0000u) +
          (double)__uint_as_float(w2 & 0xFFFF0000u);
    }
    fx_digits<NS>(x, E, u);
    fx_digits<NS>(y, E, v);
    uint16_t* q = o + (t >> 4) * Fx<NS>::ROW + 2 * (t & 15);
#pragma unroll
    for (int s = 0; s < NS; ++s) *(uint32_t*)(q + s * FX_BK) = fx_pack(u[s], v[s]);
  }
}

// ----------------------------------------------------------------------------- product
struct FxArgs {
  int m, n;                 // rows, complex columns of this panel
  int kb, kb_split;         // stages in all, per split (a multiple of FX_CHUNK)
  const int *EA, *EB;
  zd alpha, beta;
  zd* out;
  int64_t ldo;
  zd* ws;                   // split partials [split][n][m], or null (one split)
  int* err;
};

__device__ __forceinline__ void fx_store(const FxArgs& a, int64_t i, int64_t j, zd p) {
  p = a.alpha * p;
  zd* o = a.out + j * a.ldo + i;
  if (!(a.beta.x == 0.0 && a.beta.y == 0.0)) p += a.beta * (*o);
  *o = p;
}

template <int NS>
__global__ void __launch_bounds__(FX_THREADS, 1)
    k_gemm_fx(const __grid_constant__ CUtensorMap mA, const __grid_constant__ CUtensorMap mB, FxArgs args) {
  using L = Fx<NS>;
  extern __shared__ uint8_t smem_raw[];
  if (tc_given_up(args.err)) return;
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + L::STAGES * L::STAGE_BYTES);
  uint64_t* empty = full + L::STAGES;
  uint64_t* tfull = empty + L::STAGES;        // [level] MMA -> drain
  uint64_t* tempty = tfull + L::LEVELS;       // [level] drain -> MMA
  uint32_t* tslot = (uint32_t*)(tempty + L::LEVELS);
  volatile int* abort_flag = (volatile int*)(tslot + 1);
  volatile int* issued = (volatile int*)(tslot + 2);
  volatile int* consumed = (volatile int*)(tslot + 3);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.y * FX_BM, n0 = blockIdx.x * FX_BN;   // n0: real columns
  const int kb0 = blockIdx.z * args.kb_split;
  const int nk = min(args.kb_split, args.kb - kb0);
  const int nchunks = (nk + FX_CHUNK - 1) / FX_CHUNK;

  if (threadIdx.x == 0) {
    for (int q = 0; q < L::STAGES; ++q) { mbar_init(&full[q], 1); mbar_init(&empty[q], 1); }
    for (int q = 0; q < L::LEVELS; ++q) { mbar_init(&tfull[q], 1); mbar_init(&tempty[q], 8); }
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
  const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(FX_BN >> 3) << 17) |
                         ((uint32_t)(FX_BM >> 4) << 24);

  // drained sums of this thread's row and 32 columns, in units of the digit weight of level 4:
  // levels 0..4 exactly, the lower ones in FP32 (integers across all levels cost 32 registers
  // or the carries between two words, 1% of a product)
  long long hi[32];
  float lo[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) { hi[i] = 0; lo[i] = 0.f; }

  if (warp == 8) {
    if (lane == 0) {
      for (int kb = 0; kb < nk; ++kb) {
        const int st = kb % L::STAGES;
        if (kb >= L::STAGES) {
          if (!mbar_wait(&empty[st], ((kb / L::STAGES) + 1) & 1, WAIT_LIMIT, args.err)) { *abort_flag = 41; break; }
        }
        if (*abort_flag) break;
        uint8_t* sp = smem + st * L::STAGE_BYTES;
        mbar_expect_tx(&full[st], L::STAGE_BYTES);
        const int x = (kb0 + kb) * L::ROW;
#pragma unroll
        for (int q = 0; q < NS / 2; ++q) tma_load_2d(sp + q * (FX_BM * 128), &mA, &full[st], x + 64 * q, m0);
#pragma unroll
        for (int q = 0; q < NS / 2; ++q)
          tma_load_2d(sp + L::A_BYTES + q * (FX_BN * 128), &mB, &full[st], x + 64 * q, n0);
        *issued = kb + 1;
      }
    }
  } else if (warp == 9) {
    if (lane == 0) {
      bool ok = true;
      for (int kb = 0; kb < nk && ok; ++kb) {
        const int st = kb % L::STAGES, ch = kb / FX_CHUNK, in = kb % FX_CHUNK;
        if (!mbar_wait(&full[st], (kb / L::STAGES) & 1, WAIT_LIMIT, args.err)) { *abort_flag = 42; break; }
        *consumed = kb + 1;
        if (*abort_flag) break;
        tc_fence_after();
        const uint8_t* sp = smem + st * L::STAGE_BYTES;
        const uint64_t da = sw128_desc(sp), db = sw128_desc(sp + L::A_BYTES);
        const bool last = (in == FX_CHUNK - 1) || (kb == nk - 1);
#pragma unroll
        for (int lev = L::LEVELS - 1; lev >= 0; --lev) {
          if (in == 0 && ch > 0) {
            if (!mbar_wait(&tempty[lev], (ch - 1) & 1, WAIT_LIMIT, args.err)) { *abort_flag = 45; ok = false; break; }
            tc_fence_after();
          }
          const uint32_t dt = tmem + (uint32_t)(lev * FX_BN);
#pragma unroll
          for (int s = lev < NS ? 0 : lev - NS + 1; s <= (lev < NS ? lev : NS - 1); ++s) {
            // slice s of a tile: box s / 2, 64 bytes into the 128-byte rows when odd (descriptors count 16 bytes)
            const int t = lev - s;
            const uint64_t a = da + (uint64_t)(((s >> 1) * (FX_BM * 128) + (s & 1) * 64) >> 4);
            const uint64_t b = db + (uint64_t)(((t >> 1) * (FX_BN * 128) + (t & 1) * 64) >> 4);
            mma_bf16(dt, a, b, idesc, (in > 0 || s > (lev < NS ? 0 : lev - NS + 1)) ? 1u : 0u);
            mma_bf16(dt, a + 2, b + 2, idesc, 1u);
          }
          if (last) mma_commit(&tfull[lev]);
        }
        mma_commit(&empty[st]);
      }
    }
  } else {
    const int lanebase = 32 * (warp & 3), colhalf = 32 * (warp >> 2);
    bool ok = true;
    for (int ch = 0; ch < nchunks && ok; ++ch) {
#pragma unroll
      for (int lev = L::LEVELS - 1; lev >= 0; --lev) {
        bool got = mbar_wait_sleep(&tfull[lev], ch & 1, WAIT_LIMIT, args.err, 64u);
        got = __all_sync(0xffffffffu, got) && (__shfl_sync(0xffffffffu, *abort_flag, 0) == 0);
        if (!got) { if (lane == 0) atomicCAS((int*)abort_flag, 0, 44); ok = false; break; }
        tc_fence_after();
        float v[32];
        tmem_ld32(tmem + ((uint32_t)lanebase << 16) + (uint32_t)(lev * FX_BN + colhalf), v);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&tempty[lev])) : "memory");
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          if (lev > 4) lo[i] = fmaf(v[i], 1.f / (float)(1 << (8 * (lev > 4 ? lev - 4 : 0))), lo[i]);
          else hi[i] += (long long)__float2int_rn(v[i]) << (8 * (lev > 4 ? 0 : 4 - lev));
        }
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
        (void)mbar_wait(&full[kb % L::STAGES], (kb / L::STAGES) & 1, WAIT_LIMIT, &zero_flag);
    }
  } else if (warp < 8) {
    const int row = m0 + 32 * (warp & 3) + lane, j0 = (n0 + 32 * (warp >> 2)) >> 1;
    if (row < args.m) {
      const int ea = args.EA[row];
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        const int j = j0 + c;
        if (j >= args.n) break;
        const int eb = args.EB[j];
        // product of digit weights at level 4: 2^(EA - 6 + EB - 6 - 32)
        zd p;
        if (ea == FX_BAD || eb == FX_BAD) {
          p = mkz(__longlong_as_double(0x7FF8000000000000ll), __longlong_as_double(0x7FF8000000000000ll));
        } else {
          p = mkz(scalbn((double)hi[2 * c] + (double)lo[2 * c], ea + eb - 44),
                  scalbn((double)hi[2 * c + 1] + (double)lo[2 * c + 1], ea + eb - 44));
        }
        if (args.ws) args.ws[((int64_t)blockIdx.z * args.n + j) * args.m + row] = p;
        else fx_store(args, row, j, p);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u));
  }
}

__global__ void k_fx_reduce(FxArgs a, int splits) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t plane = (int64_t)a.n * a.m;
  if (t >= plane) return;
  zd sum = a.ws[t];
  for (int z = 1; z < splits; ++z) sum += a.ws[z * plane + t];
  fx_store(a, t % a.m, t / a.m, sum);
}

// ----------------------------------------------------------------------------- host
// Where the lines lie: a product of fewer complex multiply-adds than the
// slicing, product and reduction launches are worth runs on the FP64 pipe
// (about 0.9 TFLOP/s in k_zgemm_rows/cols), and so do shapes whose padding to
// 128 x 32-column tiles would be most of the work.
bool zgemm_fx_wanted(int64_t m, int64_t n, int64_t k) {
  return m >= 32 && n >= 6 && k >= 32 && (double)m * (double)n * (double)k >= 3.0e6 && k <= ((int64_t)1 << 20) &&
         m <= ((int64_t)1 << 30) && n <= ((int64_t)1 << 30);
}

#define TRY_FX(x)          \
  do {                     \
    int _r = (x);          \
    if (_r) return _r;     \
  } while (0)

struct FxPlan {
  int64_t kb, mp, np;        // stages; rows and complex columns of a panel
  size_t a_bytes, b_bytes, e_bytes, ws_bytes;
};
constexpr size_t FX_PARTIALS = (size_t)64 << 20;

static size_t fx_up(size_t b) { return (b + 255) & ~(size_t)255; }

static FxPlan fx_plan(int64_t m, int64_t n, int64_t k, size_t panel) {
  FxPlan p;
  p.kb = (2 * k + FX_BK - 1) / FX_BK;
  const size_t row = (size_t)p.kb * Fx<FX_SLICES>::ROW * 2;
  p.mp = std::max<int64_t>(FX_BM, (int64_t)(panel / row) / FX_BM * FX_BM);
  p.mp = std::min(p.mp, std::min<int64_t>(m, 65535 * FX_BM));
  p.np = std::max<int64_t>(FX_BN / 2, (int64_t)(panel / (2 * row)) / (FX_BN / 2) * (FX_BN / 2));
  p.np = std::min(p.np, n);
  p.a_bytes = fx_up(row * p.mp);
  p.b_bytes = fx_up(2 * row * p.np);
  p.e_bytes = fx_up(sizeof(int) * (size_t)(p.mp + p.np));
  p.ws_bytes = FX_PARTIALS;
  return p;
}

size_t zgemm_fx_bytes(int64_t m, int64_t n, int64_t k, size_t panel) {
  const FxPlan p = fx_plan(m, n, k, panel);
  return p.a_bytes + p.b_bytes + p.e_bytes + p.ws_bytes;
}

static FxSrc fx_src(const zd* p, int64_t si, int64_t sk, bool conj, bool dup, int64_t rows, int64_t K, int64_t kb,
                    uint16_t* d, int* e) {
  FxSrc S;
  S.p = p; S.si = si; S.sk = sk; S.conj = conj ? 1 : 0; S.dup = dup ? 1 : 0;
  S.rows = rows; S.K = K; S.kb = kb; S.d = d; S.e = e;
  S.kfast = (sk == 1) ? 1 : 0;
  const int64_t groups = S.kfast ? rows : (rows + 15) / 16;
  // long rows of a small operand are shared by several blocks (each finds the
  // row's exponent for itself) until there are two blocks per SM
  const int64_t most = std::max<int64_t>(1, kb / (S.kfast ? 16 : 4));
  S.segs = (int)std::min<int64_t>(most, std::max<int64_t>(1, 304 / std::max<int64_t>(groups, 1)));
  S.blocks = groups * S.segs;
  return S;
}

// K splits: the count of CTAs per split in whole waves of the 152 SMs, each
// split costing its stages plus about four stages of prologue and epilogue.
static int fx_splits(int64_t tiles, int64_t kb, int64_t elems) {
  const int64_t chunks = (kb + FX_CHUNK - 1) / FX_CHUNK;
  int best = 1;
  double cost = 1e300;
  for (int64_t sp = 1; sp <= std::min<int64_t>(chunks, 152); ++sp) {
    if (sp > 1 && (size_t)(sp * elems) * sizeof(zd) > FX_PARTIALS) break;
    const int64_t per = (chunks + sp - 1) / sp;
    if (per > 1024) continue;    // keeps the 64-bit sums far from overflow
    const double c = (double)((tiles * sp + 151) / 152) * (double)(per * FX_CHUNK + 4) + (sp > 1 ? 2.0 + 0.1 * sp : 0.0);
    if (c < cost) { cost = c; best = (int)sp; }
  }
  return best;
}

template <int NS>
static int fx_attributes() {
  static DeviceOnce attr;   // one instance per template instantiation
  if (!attr.need()) return 0;
  cudaError_t e = cudaFuncSetAttribute(k_gemm_fx<NS>, cudaFuncAttributeMaxDynamicSharedMemorySize, Fx<NS>::SMEM);
  if (e != cudaSuccess) { set_error(std::string("zgemm_fx: shared-memory opt-in: ") + cudaGetErrorString(e)); return 3; }
  attr.done();
  return 0;
}

// One panel: sliced operands (a.m rows of A, 2 a.n rows of B'), kb stages; part:
// FX_PARTIALS bytes.
template <int NS>
static int fx_panel(const uint16_t* da, const uint16_t* db, FxArgs a, zd* part, cudaStream_t s) {
  TRY_FX(fx_attributes<NS>());
  const int64_t ld = (int64_t)a.kb * Fx<NS>::ROW;
  CUtensorMap mA, mB;
  TRY_FX(make_map(&mA, da, a.m, ld, ld, FX_BM));
  TRY_FX(make_map(&mB, db, 2 * (int64_t)a.n, ld, ld, FX_BN));
  const int64_t mt = (a.m + FX_BM - 1) / FX_BM, nt = (2 * (int64_t)a.n + FX_BN - 1) / FX_BN;
  int sp = fx_splits(mt * nt, a.kb, (int64_t)a.m * a.n);
  const int64_t chunks = (a.kb + FX_CHUNK - 1) / FX_CHUNK, per = (chunks + sp - 1) / sp;
  sp = (int)((chunks + per - 1) / per);   // every split has work
  a.kb_split = (int)(per * FX_CHUNK);
  a.ws = sp > 1 ? part : nullptr;
  dim3 grid((unsigned)nt, (unsigned)mt, (unsigned)sp);
  k_gemm_fx<NS><<<grid, FX_THREADS, Fx<NS>::SMEM, s>>>(mA, mB, a);
  note_launch();
  if (sp > 1) {
    k_fx_reduce<<<(unsigned)(((int64_t)a.m * a.n + 255) / 256), 256, 0, s>>>(a, sp);
    note_launch();
  }
  return 0;
}

int zgemm_fx(int64_t m, int64_t n, int64_t k, zd alpha, ZView A, ZView B, zd beta, zd* C, int64_t ldc, void* ws,
             int* err, cudaStream_t s, size_t panel) {
  if (m <= 0 || n <= 0 || k <= 0) return 0;
  const FxPlan P = fx_plan(m, n, k, panel);
  char* base = (char*)ws;
  uint16_t* da = (uint16_t*)base;
  uint16_t* db = (uint16_t*)(base + P.a_bytes);
  int* ea = (int*)(base + P.a_bytes + P.b_bytes);
  int* eb = ea + P.mp;
  zd* part = (zd*)(base + P.a_bytes + P.b_bytes + P.e_bytes);
  for (int64_t j0 = 0; j0 < n; j0 += P.np) {
    const int64_t nn = std::min(P.np, n - j0);
    for (int64_t i0 = 0; i0 < m; i0 += P.mp) {
      const int64_t mm = std::min(P.mp, m - i0);
      FxSrc sa = fx_src(A.p + i0 * A.rs, A.rs, A.cs, A.conj, false, mm, k, P.kb, da, ea);
      FxSrc sb = fx_src(B.p + j0 * B.cs, B.cs, B.rs, B.conj, true, nn, k, P.kb, db, eb);
      if (i0 > 0) sb.blocks = 0;   // B' of this column panel is in place
      k_fx_slice<FX_SLICES><<<(unsigned)(sa.blocks + sb.blocks), 256, 0, s>>>(sa, sb);
      note_launch();
      FxArgs a;
      a.m = (int)mm; a.n = (int)nn;
      a.kb = (int)P.kb;
      a.EA = ea; a.EB = eb;
      a.alpha = alpha; a.beta = beta;
      a.out = C + j0 * ldc + i0;
      a.ldo = ldc;
      a.err = err;
      TRY_FX(fx_panel<FX_SLICES>(da, db, a, part, s));
    }
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { set_error(std::string("zgemm_fx: ") + cudaGetErrorString(e)); return 3; }
  return 0;
}

// ----------------------------------------------------------------------------- operators kept as slices
void fx_operand_bytes(int64_t rows, int64_t K, int64_t* kb, size_t* digits, size_t* exps) {
  *kb = (K + FX_BK - 1) / FX_BK;
  *digits = fx_up((size_t)rows * (size_t)(*kb) * Fx<FX_OP_SLICES>::ROW * 2);
  *exps = fx_up(sizeof(int) * (size_t)rows);
}

int fx_slice_planes(const uint16_t* const* planes, int nplanes, int64_t rows, int64_t K, int64_t ld,
                    const FxOperand& out, cudaStream_t s) {
  k_fx_slice_planes<FX_OP_SLICES><<<(unsigned)rows, 256, 0, s>>>(planes[0], nplanes > 1 ? planes[1] : nullptr,
                                                                 nplanes > 2 ? planes[2] : nullptr, K, ld, out.kb, out.d,
                                                                 out.e);
  note_launch();
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { set_error(std::string("fx_slice_planes: ") + cudaGetErrorString(e)); return 3; }
  return 0;
}

size_t fx_apply_bytes(int64_t n, int64_t K) {
  int64_t kb;
  size_t d, e;
  fx_operand_bytes(2 * n, K, &kb, &d, &e);
  return d + e + FX_PARTIALS;
}

int fx_apply(const FxOperand& A, int64_t m, int64_t n, int64_t k, zd alpha, const zd* X, int64_t ldx, zd beta, zd* Y,
             int64_t ldy, void* ws, int* err, cudaStream_t s) {
  if (m <= 0 || n <= 0) return 0;
  int64_t kb;
  size_t db, eb;
  fx_operand_bytes(2 * n, 2 * k, &kb, &db, &eb);
  uint16_t* d = (uint16_t*)ws;
  int* e = (int*)((char*)ws + db);
  FxSrc none{};
  FxSrc sb = fx_src(X, ldx, 1, false, true, n, k, kb, d, e);
  k_fx_slice<FX_OP_SLICES><<<(unsigned)sb.blocks, 256, 0, s>>>(none, sb);
  note_launch();
  FxArgs a;
  a.m = (int)m; a.n = (int)n;
  a.kb = (int)kb;
  a.EA = A.e; a.EB = e;
  a.alpha = alpha; a.beta = beta;
  a.out = Y;
  a.ldo = ldy;
  a.err = err;
  TRY_FX(fx_panel<FX_OP_SLICES>(A.d, d, a, (zd*)((char*)ws + db + eb), s));
  cudaError_t er = cudaGetLastError();
  if (er != cudaSuccess) { set_error(std::string("fx_apply: ") + cudaGetErrorString(er)); return 3; }
  return 0;
}

}  // namespace wcs
