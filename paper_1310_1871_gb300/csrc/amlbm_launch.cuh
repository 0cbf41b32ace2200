// Programmatic dependent launch (sm_90 and later): a kernel launched with launch_pdl
// may start while the kernel before it on the stream still runs.  It may read what
// was complete before that kernel was launched (descriptors and tile lists: whoever uploads
// them synchronises before the first launch) before pdl_wait(), everything else only after
// it: the wait returns when the kernels before it have finished and their writes are visible.
// What they write is not read through const __restrict__ kernel arguments or __ldg, which
// promise data that stays the same while this kernel runs.
// pdl_trigger() lets the next kernel of the stream start early in turn; its blocks
// take only room that this kernel's blocks, all placed by then, leave free.
//
// A timestep is one or two short kernels, so on small lattices the launch latency
// between them counts: measured on empty kernels of 152 blocks, 2.35 us per launch
// in stream order, 1.35 us with this attribute (the host's launch rate).
#pragma once

#include <cuda_runtime.h>

namespace amlbm {
namespace {

__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... K, class... A>
cudaError_t launch_pdl(void (*kernel)(K...), dim3 grid, int block, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchConfig_t c = {};
  c.gridDim = grid;
  c.blockDim = dim3((unsigned)block);
  c.dynamicSmemBytes = smem;
  c.stream = s;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &at;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, kernel, static_cast<K>(args)...);
}

}  // namespace
}  // namespace amlbm
