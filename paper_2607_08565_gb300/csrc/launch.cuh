// Kernel launches with programmatic stream serialisation.
#pragma once

#include <cuda_runtime.h>

#include <utility>

#include "smetric_impl.cuh"

namespace smetric {

// Programmatic dependent launch: a kernel launched with programmatic stream
// serialisation is set up while its predecessor still runs and waits here
// until that predecessor has finished and its writes are visible (a no-op for
// an ordinary launch). No kernel triggers its successor early: successors
// waiting on the SMs during a kernel's run measured slower.
__device__ __forceinline__ void pdl_enter() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

// Launches a kernel; with pdl the launch may begin while the previous kernel
// on the stream is still running (the kernel waits in pdl_enter).
template <typename... KArgs, typename... Args>
int launch_k(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, bool pdl,
             Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = pdl ? attr : nullptr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cuda_status(cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...));
}

}  // namespace smetric
