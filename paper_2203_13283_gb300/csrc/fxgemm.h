// Complex FP64 products on the tensor cores through fixed-point slices
// (fxgemm.cu).
#pragma once
#include "internal.h"

namespace wcs {

constexpr int FX_SLICES = 8;   // 8-bit digits per value: 63 bits below each row's largest entry

// True when zgemm_fx is the faster route for the shape (see fxgemm.cu).
bool zgemm_fx_wanted(int64_t m, int64_t n, int64_t k);
// Slices of each operand that lie in device memory at a time, at most (or one tile's).
constexpr size_t FX_PANEL = (size_t)512 << 20;
// Device workspace of one call (bounded: large operands go through in panels).
size_t zgemm_fx_bytes(int64_t m, int64_t n, int64_t k, size_t panel = FX_PANEL);
// C (m x n, column-major ldc) = alpha * A (m x k) * B (k x n) + beta * C, each entry
// to k max |A_i.| max |B_.j| 2^-55 and the rounding of the result (see fxgemm.cu).  ws: zgemm_fx_bytes of device memory; err:
// device flag of the bounded waits (zero before the first use).  C must not
// overlap A or B.
int zgemm_fx(int64_t m, int64_t n, int64_t k, zd alpha, ZView A, ZView B, zd beta, zd* C, int64_t ldc, void* ws,
             int* err, cudaStream_t s, size_t panel = FX_PANEL);

// The mixed form's operators for exact residuals: rows kept as six digits (47 bits
// below each row's largest entry; their entries carry 24) plus an exponent.
constexpr int FX_OP_SLICES = 6;
struct FxOperand {
  uint16_t* d = nullptr;   // [row][kb][FX_OP_SLICES][32]
  int* e = nullptr;        // exponent per row
  int64_t kb = 0;
};
// Stages and bytes (digits, exponents; 256-byte multiples) of rows x K real values.
void fx_operand_bytes(int64_t rows, int64_t K, int64_t* kb, size_t* digits, size_t* exps);
// Slices of split-bf16 planes (row-major, ld values a row).
int fx_slice_planes(const uint16_t* const* planes, int nplanes, int64_t rows, int64_t K, int64_t ld,
                    const FxOperand& out, cudaStream_t s);
// Y (m x n, ldy) = alpha * A X + beta * Y for a sliced A (m x k complex) and FP64
// X (k x n, ldx), X as six digits below each column's largest entry: errors of 2^-47 of
// the column's and the row's largest entries a term, and the rounding of the result.  ws: fx_apply_bytes(n, 2 k).
size_t fx_apply_bytes(int64_t n, int64_t K);
int fx_apply(const FxOperand& A, int64_t m, int64_t n, int64_t k, zd alpha, const zd* X, int64_t ldx, zd beta, zd* Y,
             int64_t ldy, void* ws, int* err, cudaStream_t s);

}  // namespace wcs
