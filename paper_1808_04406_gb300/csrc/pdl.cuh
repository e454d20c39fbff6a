// Programmatic dependent launch: a kernel of a chain of steps is launched while its
// predecessor still runs, so that launch latency, block scheduling and the first
// instruction fetches overlap with the predecessor's last blocks; chain_wait()
// then waits until the predecessor has completed and its stores are visible.
// Every kernel of the chain waits before it touches the populations, so one that
// has completed implies all earlier ones have.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace lbm {

__device__ __forceinline__ void chain_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // only now: released before the wait, kernels further down the chain would pile up
  // on the SMs and unbalance them (FP64 128^2: 58 us a step instead of 21)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... P, typename... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, A&&... args) {
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, P(std::forward<A>(args))...);
}

}  // namespace lbm
