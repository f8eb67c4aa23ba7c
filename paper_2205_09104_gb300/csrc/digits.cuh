// FP64 stencil on the tensor cores by exact digit products (digits.cu): operand layouts and launchers.
#pragma once

#include "common.cuh"

namespace coarse {

constexpr int kDigCols = 2;  // columns of one pass

// Halves of the packed digits of one (column, site): [part][digit][n]; bytes of one record of row
// corrections: [sigma3 variant][part][level] floats.
__host__ __device__ constexpr size_t dig_x_halves(int n) { return 16 * (size_t)n; }
constexpr size_t kDigCorr = 32;

// Bytes of the column operands of `cols` columns on V sites: digits, corrections, scales.
__host__ __device__ inline size_t dig_x_bytes(int n, int V, int cols) {
  return (size_t)cols * V * (dig_x_halves(n) * 2 + kDigCorr * sizeof(float) + sizeof(double));
}

// Blocks of one operator as digits and their scales (sizes: dig_block_bytes, dig_scale_bytes).
inline size_t dig_block_bytes(int n, int V) { return (size_t)V * 5 * n * n * 16; }
inline size_t dig_scale_bytes(int V) { return (size_t)V * 5 * sizeof(double); }
int launch_dig_blocks(const double2* blocks, int V, int n, void* dig, double* scale, cudaStream_t s);

// y = D x (with a's epilogue) for ncol <= kDigCols columns x + c * ldc, y + c * ldc, through the digit
// operands a.dig (must be set); a.digx holds room for ncol columns.
int launch_apply_digits(int n, const ApplyArgs& a, int ncol, long long ldc, cudaStream_t s);

}  // namespace coarse
