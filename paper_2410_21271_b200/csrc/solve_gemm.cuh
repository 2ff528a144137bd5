// The fp32 products of the offline solve on the 5th-generation tensor cores (solve_gemm.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace eora {

// An operand of split_gemm: rows x cols fp32 values (both multiples of 128, cols being the reduction axis) as three bf16 numbers each,
// in blocks of 128 rows x 32 columns: [row block][column block][plane][128 rows][64 bytes], the 16-byte pieces of a row in the order of
// the 64-byte swizzle of a K-major operand, so that a plane of a block is one 8 KB copy into shared memory.
constexpr int kSplitRows = 128, kSplitCols = 32, kSplitPlane = kSplitRows * kSplitCols * 2, kSplitBlock = 3 * kSplitPlane;
inline size_t split_bytes(int rows, int cols) { return (size_t)(rows / kSplitRows) * (cols / kSplitCols) * kSplitBlock; }

// out (may be null) = split(a - b) (b may be null) of [rows][cols] fp32, leading dimension lda, padded with zeros to rows_p x cols_p.  copy
// (may be null): a - b itself, padded, as [rows_p][cols_p] fp32, rows ld_copy apart.
cudaError_t split_rows(cudaStream_t st, const float* a, const float* b, int rows, int cols, int lda, int rows_p, int cols_p, uint8_t* out, float* copy,
                       int ld_copy);
// out = split(a^T): a is [rows][cols] fp32, the operand has cols_p rows and rows_p columns.  copy (may be null): a, padded, as [rows_p][cols_p].
cudaError_t split_cols(cudaStream_t st, const float* a, int rows, int cols, int lda, int rows_p, int cols_p, uint8_t* out, float* copy = nullptr);

// C [m][ldc] = A B^T with A [m][k] and B [n][k] split as above; m, n, k multiples of 128.  sym: A and B are the same operand, and only tiles
// on and below the diagonal are computed and stored to both places.  add: C += instead.  status: not zero if a wait inside the kernel ran out.
cudaError_t split_gemm(cudaStream_t st, const uint8_t* a, const uint8_t* b, int m, int n, int k, float* c, int ldc, bool sym, bool add, int sm_count,
                       int* status);

// The same for B with n (a multiple of `width`: 64, 96, 128 or 160) rows, split as a matrix of whole blocks: C [m][ldc] = A B^T - *shift Y
// (shift, Y [m][ldc]: may be null; Y must not be C).
cudaError_t split_skinny(cudaStream_t st, int width, const uint8_t* a, const uint8_t* b, int m, int n, int k, float* c, int ldc, const float* y,
                         const float* shift, int* status);

}  // namespace eora
