// Bookkeeping of the digit copies (dig_store.cuh); no device code.
#include "dig_store.cuh"

#include <algorithm>
#include <mutex>
#include <utility>
#include <vector>

#include "../../include/coarse.h"

namespace coarse {

struct DigStore {
  std::mutex mu;
  int device = 0;
  bool off = false;      // asked for at creation
  bool refused = false;  // no room, or given back
  bool kept = false;     // a captured graph holds the pointers
  int users = 0;         // calls that are launching with the pointers
  void* dig = nullptr;
  double* scale = nullptr;
  void* work = nullptr;
  size_t bytes = 0;
};

namespace {

// The live stores, and the bytes of their copies by device.  Lock order: a store's mutex, then this one; the other way
// round only by try_lock.
std::mutex g_mu;
std::vector<DigStore*> g_stores;
constexpr int kDevices = 64;
size_t g_bytes[kDevices];

bool reserve(int dev, size_t bytes) {
  size_t mfree = 0, total = 0;
  if (dev < 0 || dev >= kDevices || cudaMemGetInfo(&mfree, &total) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  std::lock_guard<std::mutex> lk(g_mu);
  if (g_bytes[dev] + bytes > total / 4) return false;
  g_bytes[dev] += bytes;
  return true;
}

void unreserve(int dev, size_t bytes) {
  std::lock_guard<std::mutex> lk(g_mu);
  g_bytes[dev] -= bytes;
}

void free_copy(DigStore* st) {
  cudaFree(st->dig);
  cudaFree(st->scale);
  cudaFree(st->work);
  st->dig = st->work = nullptr;
  st->scale = nullptr;
}

template <class T>
bool take(T** p, size_t bytes) {
  if (cudaMalloc((void**)p, bytes) == cudaSuccess) return true;
  cudaGetLastError();
  *p = nullptr;
  return false;
}

bool capturing(cudaStream_t s) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &cap) == cudaSuccess) return cap != cudaStreamCaptureStatusNone;
  cudaGetLastError();  // the legacy stream while another one is captured
  return true;
}

// Allocations of this thread do not disturb a capture of another stream (they are not part of it).
struct RelaxedCapture {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
  ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

// Gives the copies of the current device back that nothing uses; false if there was none.
bool reclaim() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  std::lock_guard<std::mutex> lk(g_mu);
  std::vector<std::pair<DigStore*, std::unique_lock<std::mutex>>> idle;
  for (DigStore* st : g_stores) {
    std::unique_lock<std::mutex> own(st->mu, std::try_to_lock);
    if (own && st->device == dev && st->dig && st->users == 0 && !st->kept) idle.emplace_back(st, std::move(own));
  }
  if (idle.empty()) return false;
  // kernels that still read a copy end first (no call can start another: the locks are held); an error if a stream
  // is being captured in a mode that forbids it
  if (cudaDeviceSynchronize() != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  for (auto& it : idle) {
    free_copy(it.first);
    it.first->refused = true;
    g_bytes[dev] -= it.first->bytes;
  }
  return true;
}

}  // namespace

DigStore* dig_store_new(int device, bool off) {
  DigStore* st = new DigStore();
  st->device = device;
  st->off = off;
  std::lock_guard<std::mutex> lk(g_mu);
  g_stores.push_back(st);
  return st;
}

void dig_store_delete(DigStore* st) {
  if (!st) return;
  {
    std::lock_guard<std::mutex> lk(g_mu);
    g_stores.erase(std::remove(g_stores.begin(), g_stores.end(), st), g_stores.end());
    if (st->dig) g_bytes[st->device] -= st->bytes;
  }
  if (st->dig) free_copy(st);
  delete st;
}

void dig_store_retry(DigStore* st) {
  std::lock_guard<std::mutex> lk(st->mu);
  st->refused = false;
}

int dig_store_path(DigStore* st) {
  std::lock_guard<std::mutex> lk(st->mu);
  return st->dig ? COARSE_FP64_DIGITS : st->off ? COARSE_FP64_PIPE_ASKED : st->refused ? COARSE_FP64_PIPE_MEMORY
                                                                                    : COARSE_FP64_UNDECIDED;
}

int dig_store_refill(DigStore* st, const DigPlan& plan, cudaStream_t s) {
  std::lock_guard<std::mutex> lk(st->mu);
  return st->dig ? plan.pack(plan.ctx, st->dig, st->scale, s) : COARSE_OK;
}

DigUse::DigUse(DigStore* st, const DigPlan& plan, cudaStream_t s) {
  std::lock_guard<std::mutex> lk(st->mu);
  if (st->off || (st->refused && !st->dig)) return;
  const bool cap = capturing(s);
  if (!st->dig) {
    if (cap) return;  // nothing can be allocated
    const RelaxedCapture relaxed;
    st->bytes = plan.dig + plan.scale + plan.work;
    if (!reserve(st->device, st->bytes)) {
      st->refused = true;
      return;
    }
    if (!take(&st->dig, plan.dig) || !take(&st->scale, plan.scale) || !take(&st->work, plan.work)) {
      free_copy(st);
      unreserve(st->device, st->bytes);
      st->refused = true;
      return;
    }
    rc_ = plan.pack(plan.ctx, st->dig, st->scale, s);
    // once: calls on other streams may follow without waiting for this one's
    if (rc_ == COARSE_OK && cudaStreamSynchronize(s) != cudaSuccess) rc_ = COARSE_ERR_CUDA;
    if (rc_ != COARSE_OK) {
      free_copy(st);
      unreserve(st->device, st->bytes);
      st->refused = true;
      return;
    }
  }
  if (cap) st->kept = true;
  ++st->users;
  st_ = st;
  dig_ = st->dig;
  scale_ = st->scale;
  work_ = st->work;
}

DigUse::~DigUse() {
  if (!st_) return;
  std::lock_guard<std::mutex> lk(st_->mu);
  --st_->users;
}

cudaError_t device_malloc(void** p, size_t bytes) {
  cudaError_t e = cudaMalloc(p, bytes);
  if (e != cudaErrorMemoryAllocation) return e;
  cudaGetLastError();
  return reclaim() ? cudaMalloc(p, bytes) : e;
}

}  // namespace coarse
