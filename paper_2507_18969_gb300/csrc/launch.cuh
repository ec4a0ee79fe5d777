// Kernel launch with programmatic dependent launch (PDL).
//
// Every kernel of the step is launched with programmatic stream
// serialisation, so the next kernel on the stream is scheduled while the
// current one finishes. Each kernel therefore starts with pdl_wait(), which
// returns once the preceding grid has completed and its writes are visible,
// and then calls pdl_launch() to let its own successor be scheduled. A
// kernel launched without the attribute treats both as no-ops.
#pragma once

#include <cuda_runtime.h>

#include <utility>

#include "once.cuh"

namespace edpc {

// f (kernel attributes, ...) once on the current device.
template <class F>
inline cudaError_t once_on_device(OncePerDevice& once, F&& f) {
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  return e != cudaSuccess ? e : once.run(dev, f);
}

// The current device's SM count (at least 1).
inline cudaError_t sm_count(int* n) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(n, cudaDevAttrMultiProcessorCount, dev);
  return e;
}

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Launches from the calling thread use the PDL attribute while this is true.
inline thread_local bool g_pdl_enabled = true;

// Turns the PDL attribute off for the launches made in its scope (kernels whose
// stream also waits on an event, i.e. with more than one incoming dependency).
struct NoPdl {
  bool saved;
  NoPdl() : saved(g_pdl_enabled) { g_pdl_enabled = false; }
  ~NoPdl() { g_pdl_enabled = saved; }
};

// Keeps the attribute as it is when `on`, else turns it off for the scope.
struct PdlScope {
  bool saved;
  explicit PdlScope(bool on) : saved(g_pdl_enabled) { g_pdl_enabled = saved && on; }
  ~PdlScope() { g_pdl_enabled = saved; }
};

template <typename... KArgs, typename... Args>
inline cudaError_t launch_k(void (*k)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                            Args&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = g_pdl_enabled ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k, std::forward<Args>(args)...);
}

}  // namespace edpc
