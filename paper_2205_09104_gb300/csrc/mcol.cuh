// Multi-column stencil and half apply (mcol.cu).
#pragma once

#include "batch.cuh"
#include "common.cuh"

namespace coarse {

constexpr int kMcCols = 12;  // columns of one pass (shared memory holds their vectors)

// y = D x for R <= kMcCols complex64 columns (x + c * ldc -> y + c * ldc) on the FP32 blocks of `a`, plain
// epilogue; x 16-byte aligned, ldc even.
int launch_apply_mc(int n, const ApplyArgs& a, int R, long long ldc, cudaStream_t s);

// The batched phases (half apply, full stencil) over the items of one n-group.
int launch_beo_mc(int prec, int n, const McPhase& p, cudaStream_t s);
int launch_bapply_mc(int prec, int n, const McPhase& p, cudaStream_t s);

}  // namespace coarse
