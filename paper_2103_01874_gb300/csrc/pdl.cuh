// Programmatic dependent launch of the projection's kernel chain.
//
// Each kernel of the step is launched with programmatic stream serialisation
// and begins with pdl_enter(): griddepcontrol.wait blocks until the preceding
// kernel has completed and its memory operations are visible, so no global
// data is read before it.  No kernel signals its dependents early: the implicit
// trigger when its CTAs exit lets the next kernel's launch overlap the end of
// this one and its memory flush, which is most of a launch's cost (chain of
// small kernels: 1.4 against 4.1 us each).  An explicit trigger at the start
// (griddepcontrol.launch_dependents) packed the next kernel's CTAs into the few
// SM slots free at that moment, under the running kernel's shared-memory
// carve-out: few CTAs ended up several to an SM, and passes with many loads in
// flight kept a small L1 (128^3: 222 -> 205 us without it, 64^3 FP64 81 -> 65,
// 96^3 153 -> 144, 256^3 FP64 1238 -> 1206).  Captured launches take the same
// attribute (64-grid batch 3960 -> 3930 us, 32^3's refinement graph 74 -> 72).
#pragma once
#include <cuda_runtime.h>

#include <utility>

namespace ppe {

__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// kernel<<<grid, block, smem, st>>>(args...), with programmatic stream
// serialisation (in a capture: a programmatic edge); returns the launch's error.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                       Args&&... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

}  // namespace ppe
