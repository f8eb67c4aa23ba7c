// Host build of csrc/dig_store.cu against a fake of the runtime calls it makes (a device with a given amount of
// memory, streams that may be captured), used only by tests/test_dig_store_host.py.
#include <cuda_runtime.h>

#include <map>

static size_t g_total = 0, g_used = 0;
static int g_device = 0, g_capturing = 0, g_packs = 0, g_sync_fails = 0;
static std::map<void*, size_t> g_live;
static char* g_next = reinterpret_cast<char*>(0x1000);

extern "C" {
cudaError_t CUDARTAPI cudaMalloc(void** p, size_t bytes) {
  if (g_used + bytes > g_total) return cudaErrorMemoryAllocation;
  g_used += bytes;
  *p = g_next;
  g_next += 256;
  g_live[*p] = bytes;
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaFree(void* p) {
  if (!p) return cudaSuccess;
  g_used -= g_live.at(p);
  g_live.erase(p);
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaMemGetInfo(size_t* f, size_t* t) {
  *f = g_total - g_used;
  *t = g_total;
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  *s = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode*) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaDeviceSynchronize() { return g_sync_fails ? cudaErrorStreamCaptureUnsupported : cudaSuccess; }
cudaError_t CUDARTAPI cudaGetLastError() { return cudaSuccess; }
cudaError_t CUDARTAPI cudaGetDevice(int* d) {
  *d = g_device;
  return cudaSuccess;
}
}

#include "../paper_2205_09104_gb300/csrc/dig_store.cu"

using namespace coarse;

static DigPlan plan_of(size_t bytes) {
  DigPlan p;
  p.dig = bytes - 20;
  p.scale = 10;
  p.work = 10;
  p.ctx = nullptr;
  p.pack = [](const void*, void*, double*, cudaStream_t) {
    ++g_packs;
    return 0;
  };
  return p;
}

extern "C" {
void host_device(size_t total, int capturing, int device, int sync_fails) {
  g_total = total;
  g_capturing = capturing;
  g_device = device;
  g_sync_fails = sync_fails;
}
size_t host_used() { return g_used; }
int host_packs() { return g_packs; }
void* host_store(int device, int off) { return dig_store_new(device, off != 0); }
void host_delete(void* st) { dig_store_delete(static_cast<DigStore*>(st)); }
void host_retry(void* st) { dig_store_retry(static_cast<DigStore*>(st)); }
int host_refill(void* st, size_t bytes) { return dig_store_refill(static_cast<DigStore*>(st), plan_of(bytes), nullptr); }
int host_path(void* st) { return dig_store_path(static_cast<DigStore*>(st)); }
// a call that runs for as long as the handle lives
void* host_use(void* st, size_t bytes) { return new DigUse(static_cast<DigStore*>(st), plan_of(bytes), nullptr); }
int host_has(void* use) { return static_cast<DigUse*>(use)->dig() != nullptr; }
void host_done(void* use) { delete static_cast<DigUse*>(use); }
// 1 if an allocation of the library succeeds (it is kept)
int host_alloc(size_t bytes) {
  void* p = nullptr;
  return device_malloc(&p, bytes) == cudaSuccess;
}
}
