// The digit copy of an operator's FP64 blocks: built on the first FP64 stencil, given back when memory is short.
//
// The copy is as large as the FP64 blocks, and an operator that is only applied in FP32 or BF16 never needs it.  So
// it is built by the first FP64 stencil that is not being captured, if the copies of all operators of the device stay
// below a quarter of its memory, and the FP64 pipe serves where there is none.  Every allocation of the library goes
// through device_malloc: if one fails, the copies that no call and no captured graph is using are given back and it
// is tried again, so that whatever fits without digits still fits.  A copy that could not be built or was given back
// is not tried again before the operator's blocks change.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>

namespace coarse {

struct DigStore;

// off: never build a copy
DigStore* dig_store_new(int device, bool off);
void dig_store_delete(DigStore* st);  // no call on the operator may be in flight
// The blocks have changed: a copy that was refused or given back may be tried again.
void dig_store_retry(DigStore* st);
// Which way FP64 stencils go (coarse_fp64_path)
int dig_store_path(DigStore* st);

// What a copy takes and how it is filled from the operator (on the stream; a coarse_status).
struct DigPlan {
  size_t dig, scale, work;
  int (*pack)(const void* ctx, void* dig, double* scale, cudaStream_t s);
  const void* ctx;
};

// The copy for the duration of a call (or of a captured graph, if `s` is being captured: it is then kept for the
// operator's lifetime).  dig() is null where the FP64 pipe has to do.
class DigUse {
 public:
  DigUse(DigStore* st, const DigPlan& plan, cudaStream_t s);
  ~DigUse();
  DigUse(const DigUse&) = delete;
  DigUse& operator=(const DigUse&) = delete;
  const void* dig() const { return dig_; }
  const double* scale() const { return scale_; }
  void* work() const { return work_; }
  int rc() const { return rc_; }  // status of filling the copy

 private:
  DigStore* st_ = nullptr;
  const void* dig_ = nullptr;
  const double* scale_ = nullptr;
  void* work_ = nullptr;
  int rc_ = 0;
};
// Fills an existing copy again (the blocks have changed).
int dig_store_refill(DigStore* st, const DigPlan& plan, cudaStream_t s);

// cudaMalloc that gives unused digit copies of the current device back before it fails.
cudaError_t device_malloc(void** p, size_t bytes);

}  // namespace coarse
