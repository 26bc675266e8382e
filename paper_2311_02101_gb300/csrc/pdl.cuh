// Programmatic dependent launch: a kernel may start while its predecessor in
// the stream finishes, sets itself up from data that no kernel in flight
// writes (formula, tables), and waits for the predecessor's results before it
// touches them. Every block of such a kernel waits, so a finished kernel means
// that all before it are finished too. What a predecessor or the caller's work
// before it writes is read by plain loads after the wait, never by __ldg or
// through a const __restrict__ parameter: read-only loads are for data that does
// not change while the kernel is in flight (formula, tables, weights), and may
// be moved across the wait.
#pragma once

#include <cuda_runtime.h>

namespace rbmsat {

// the predecessor's writes are visible from here on
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// the next launch may start. After pdl_wait: at most two launches are in flight.
__device__ __forceinline__ void pdl_release() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... Params, typename... Args>
cudaError_t launch_pdl(void (*kern)(Params...), dim3 grid, int threads, int smem, cudaStream_t st,
                       const Args&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

}  // namespace rbmsat
