// Complex FP64 products on the tensor cores through fixed-point slices
// (fxgemm.cu).
#pragma once
#include "internal.h"

namespace wcs {

constexpr int FX_SLICES = 8;   // 8-bit digits per value: 63 bits below each row's largest entry

// True when zgemm_fx is the faster route for the shape (see fxgemm.cu).
bool zgemm_fx_wanted(int64_t m, int64_t n, int64_t k);
// Device workspace of one call (bounded: large operands go through in panels).
size_t zgemm_fx_bytes(int64_t m, int64_t n, int64_t k);
// C (m x n, column-major ldc) = alpha * A (m x k) * B (k x n) + beta * C, with
// the accuracy of an FP64 product.  ws: zgemm_fx_bytes of device memory; err:
// device flag of the bounded waits (zero before the first use).  C must not
// overlap A or B.
int zgemm_fx(int64_t m, int64_t n, int64_t k, zd alpha, ZView A, ZView B, zd beta, zd* C, int64_t ldc, void* ws,
             int* err, cudaStream_t s);

}  // namespace wcs
