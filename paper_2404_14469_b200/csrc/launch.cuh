// Kernel launches with programmatic dependent launch: a kernel launched this way may become
// resident while the previous kernel of the stream is still running, which hides its launch
// latency and prologue.  A kernel launched this way calls pdl_wait() before its first access
// to global memory (it returns once the previous kernel has completed and its writes are
// visible).  One does so later: the second of two select launches of a ragged batch, which runs beside the
// first.  It may because every CTA of the first has called pdl_wait() when it starts, because it takes
// what was visible to the first over by an acquire of a flag that the first released (or else waits), and
// because all its CTAs call pdl_wait() before they end: a kernel behind it that waits for it has then
// waited for the first one too (pool_topk_cluster_kernel).  A kernel that calls pdl_launch_dependents() lets the next one in early; without it
// the next one is let in when the kernel ends, which still saves most of the launch latency (the
// select kernel behind the scoring kernel starts 2.5 us earlier than with a plain launch).
// Apart from that pair only the small kernels in front of the scoring kernel let it in early (202 instead of 207 us per
// layer on the 32K GQA workload, 93 instead of 97 us on the 16K MHA one).  The scoring kernel does
// not let the select kernel in: CTAs that wait on the SMs that come free first cost 1-2 us; nor
// the select kernel the gather kernel, whose blocks would crowd there (68 instead of 60 us).
#pragma once
#include <cuda_runtime.h>

namespace snapkv {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                       cudaStream_t stream, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

}  // namespace snapkv
