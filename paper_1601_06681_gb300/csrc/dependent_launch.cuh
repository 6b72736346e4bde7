// Programmatic dependent launch for the short kernels of an iteration, each of
// which reads what the one before it wrote. A kernel launched by
// launch_dependent may start while its predecessor in the stream (or graph)
// still runs: it stages what no kernel of a step writes (operator rows, face
// ids), then dep_wait() returns once the predecessor has ended and its writes
// are visible. dep_trigger() lets the successor start in turn; a successor's
// blocks never take the place of this kernel's, which have all started then.
// Every thread that touches a step's data calls dep_wait() first, so a kernel
// ends only after its predecessor and the order of the stream is kept; after an
// ordinary launch both calls do nothing. The steady solve of 160 x 160, p = 4 with
// BF16 corrections (about 870 launches of 9 us, each a chain of four dependent
// loads before its first product) went from 8.15 to 7.15 ms.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace ehdg {

__device__ __forceinline__ void dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void dep_trigger() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <class... P, class... A>
cudaError_t launch_dependent(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                             cudaStream_t s, A&&... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

}  // namespace ehdg
