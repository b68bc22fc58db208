// Exact (fixed-point sliced) operator products for the refinement residual
// of the mixed form (exact.cu).
#pragma once
#include "internal.h"

namespace wcs {

constexpr int EX_SLICES = 6;      // 7-bit slices per value (43 bits below each chunk's scale)
constexpr int EX_CHUNK = 1024;    // K elements per scale chunk and per split of the contraction
constexpr int EX_LEVELS = 6;      // slice pairs (s, t) with s + t < EX_LEVELS are formed

// A K-major real operand (rows x K, leading dimension ld) as EX_SLICES bf16
// planes of integers plus a power-of-two exponent per (row, chunk); for a
// right-hand block the exponent is stored once per complex column (rows 2j
// and 2j + 1 of the real view share it).
struct ExactOperand {
  uint16_t* slice[EX_SLICES] = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
  int64_t ld = 0;
  int16_t* expo = nullptr;
  int64_t nchunks = 0;
};

// Leading dimension, chunk count and bytes of one slice plane and of the
// exponent table for `rows` rows of K values.
int exact_operand_alloc_bytes(int64_t rows, int64_t K, int64_t* ld, int64_t* nchunks, size_t* slice_bytes,
                              size_t* expo_bytes);
// Real rows (rows x K, row-major FP64, ld) as slices; and the exact real
// product D (M x Nc, row-major FP64, ldd) = A B^T (ws: nchunks * Nc * M floats).
int exact_slice_real(const double* X, int64_t rows, int64_t K, int64_t ld, const ExactOperand& out, cudaStream_t s);
int exact_product_real(const ExactOperand& A, int M, const ExactOperand& B, int Nc, int K, double* D, int64_t ldd,
                       float* ws, int64_t ws_elems, int* err, cudaStream_t s);

}  // namespace wcs
