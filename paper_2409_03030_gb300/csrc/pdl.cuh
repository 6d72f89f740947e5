// Programmatic dependent launch (sm_90 and later) for the kernels of the CG
// iteration chain.  Each such kernel calls pdl_enter(), or pdl_wait(), before it
// touches memory: griddepcontrol.wait returns once the preceding grid in the stream
// has completed and its writes are visible, so the kernel observes exactly
// what plain stream order would give it; it then (pdl_enter) or near its end
// (pdl_trigger) lets its own successor be launched, whose blocks take the SM slots freed by this grid's last wave and
// wait there.  What overlaps is the launch and block-scheduling ramp of each
// kernel, not any computation.  For a launch without the attribute both
// instructions have no effect.
#pragma once
#include <cuda_runtime.h>

namespace jqcd {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_enter() {
  pdl_wait();
  pdl_trigger();
}
// The kernels of 16-site tiles (eight threads per site) trigger after their main
// work instead: triggered at once, the next grid's blocks take the free slots
// of SMs that still run this one, so some SMs can end up with more of its blocks
// than others and the whole grid waits for those.  Measured on GB300 with the
// double-word tiles, trigger first against last: solve at 8^4 1.43 and 1.385 ms
// (though one hop alone, back to back, 2.31 and 2.72 us), 14^4 equal (2.92 ms).

// kern<<<grid, block, smem, s>>>(args...) with programmatic stream
// serialization allowed; kern must call pdl_enter() or pdl_wait() first.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                       Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

}  // namespace jqcd
