// FP64 stencil on the tensor cores by exact digit products (digits.cu): operand layouts and launchers.
#pragma once

#include "common.cuh"

namespace coarse {

constexpr int kDigCols = 2;  // columns of one pass

// Halves of the packed digits of one (column, site): [part][digit][n], then the magnitudes of the leading digits
// |re| + |im|, [n]; bytes of one record of row
// corrections: [sigma3 variant][part][level] floats.
__host__ __device__ constexpr size_t dig_x_halves(int n) { return 17 * (size_t)n; }
constexpr size_t kDigCorr = 32;

// Bytes of the column operands of `cols` columns on V sites: digits, corrections, scales, the rows' demands.
__host__ __device__ inline size_t dig_x_bytes(int n, int V, int cols) {
  return (size_t)cols * V * (dig_x_halves(n) * 2 + kDigCorr * sizeof(float) + sizeof(double) + sizeof(float));
}
// Bytes of the work memory of a stencil of up to `cols` columns per pass: the column operands, behind
// those of one column the push kernel's row magnitudes and exponents.
inline size_t dig_work_bytes(int n, int V, int cols) {
  const size_t push = dig_x_bytes(n, V, 1) + (size_t)5 * V * (n * sizeof(float) + sizeof(int));
  const size_t pass = dig_x_bytes(n, V, cols);
  return push > pass ? push : pass;
}

// Blocks of one operator as digits and their scales (sizes: dig_block_bytes, dig_scale_bytes).
inline size_t dig_block_bytes(int n, int V) { return (size_t)V * 5 * n * n * 16; }
inline size_t dig_scale_bytes(int V) { return (size_t)V * 5 * sizeof(double); }
int launch_dig_blocks(const double2* blocks, int V, int n, void* dig, double* scale, cudaStream_t s);

// Columns that one pass of a multi-column FP64 stencil should take (1 or kDigCols).
int dig_columns(int n, int V);
// How the copy of `op` is built (up to `op->max_nrhs` columns a call).
DigPlan dig_plan(const coarse_op* op);
// y = D x (with a's epilogue) for ncol <= kDigCols columns x + c * ldc, y + c * ldc, through the operator's digits
// (d.dig() must be set).
int launch_apply_digits(int n, const ApplyArgs& a, const DigUse& d, int ncol, long long ldc, cudaStream_t s);
// y = D x (with a's epilogue), one column, in FP64: through the operator's digits, or on the FP64 pipe.
int launch_apply64(const coarse_op* op, const ApplyArgs& a, cudaStream_t s);

// Batched FP64 residual: one pass = up to kDigCols columns of one operator.  Launches cover the passes' sites
// padded to kDigMapSites each; map[i] is the pass of sites i * kDigMapSites ..
constexpr int kDigMapSites = 64;
struct DigPass {
  const double2* x;  // columns at x + c ldx, addends z + c ldx, results y + c ldy
  const double2* z;
  double2* y;
  size_t ldx, ldy;
  const void* dig;
  const double* digscale;
  void* digx;        // room for `cols` columns
  const void* blocks;
  const int* nb;
  double mu;
  int V, cols;
  int start;         // first site of the pass in the launch
  int q0;            // first solve
};
// r = b - D x of the passes with a column that is not done (flags[2 q + 1]); sites: a multiple of kDigMapSites
int launch_bresidual_digits(int n, const DigPass* passes, const int* map, int sites, const int* flags,
                            const double2* coef, cudaStream_t s);

}  // namespace coarse
