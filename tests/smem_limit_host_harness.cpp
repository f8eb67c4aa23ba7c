// Host build of csrc/smem_limit.cuh against a fake of the two runtime calls it makes, used only by
// tests/test_smem_limit_host.py.
#include <cuda_runtime.h>

static int g_device = 0, g_fail = 0, g_calls = 0, g_bytes = 0;

extern "C" cudaError_t CUDARTAPI cudaGetDevice(int* dev) {
  *dev = g_device;
  return cudaSuccess;
}
extern "C" cudaError_t CUDARTAPI cudaFuncSetAttribute(const void*, cudaFuncAttribute, int value) {
  ++g_calls;
  g_bytes = value;
  return g_fail ? cudaErrorInvalidValue : cudaSuccess;
}

#include "../paper_2205_09104_gb300/csrc/smem_limit.cuh"

static coarse::SmemLimit g_limit;

extern "C" {

// Raises the limit on device `dev`; returns the status, *calls receives the attribute calls made so far.
int host_raise(int dev, int bytes, int fail, int* calls, int* last) {
  g_device = dev;
  g_fail = fail;
  const int rc = (int)coarse::raise_smem_limit(g_limit, nullptr, (size_t)bytes);
  *calls = g_calls;
  *last = g_bytes;
  return rc;
}

}  // extern "C"
