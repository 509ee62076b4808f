// Status flags of the tensor-core kernels.  Every tcgen05 kernel bounds its
// mbarrier waits; one that gives up sets its translation unit's device flag
// (the split-TF32 product's in tc32.cu, the emulated-FP64 one's in ozaki.cu),
// and the library reads and clears them after the launches of an API call
// (HS_ETIMEOUT).  The flag defined here is the one a test raises from the host.
#include <atomic>

#include "linalg.cuh"

namespace hs {

// Raised from the host by the failure-injection hook (hs_raise_tc_timeout).
__device__ int g_tc_timeout = 0;

// Set the current device's timeout flag from the host (test hook: the next
// call that checks it reports HS_ETIMEOUT; no kernel waits on anything).
static std::atomic<bool> g_raised{false};

cudaError_t tc_raise_timeout_flag() {
  const int one = 1;
  const cudaError_t e = cudaMemcpyToSymbol(g_tc_timeout, &one, sizeof(int), 0, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) g_raised = true;
  return e;
}

bool tc_timeout_raised() { return g_raised; }

bool tc_timed_out(cudaStream_t s) {
  int v[3] = {0, 0, 0};
  cudaMemcpyFromSymbolAsync(&v[0], g_tc_timeout, sizeof(int), 0, cudaMemcpyDeviceToHost, s);
  oz_timeout_flag(s, &v[1], false);
  t32_timeout_flag(s, &v[2], false);
  cudaStreamSynchronize(s);
  const bool out = v[0] || v[1] || v[2];
  if (out) {
    if (v[0]) g_raised = false;
    v[0] = 0;
    cudaMemcpyToSymbolAsync(g_tc_timeout, v, sizeof(int), 0, cudaMemcpyHostToDevice, s);
    oz_timeout_flag(s, v, true);
    t32_timeout_flag(s, v, true);
    cudaStreamSynchronize(s);
  }
  return out;
}

}  // namespace hs
