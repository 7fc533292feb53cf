// The launch of a step kernel, with or without programmatic stream serialisation.
#pragma once

#include <cuda_runtime.h>

namespace lbm {

// Step kernels begin with step_grid_enter; launched with programmatic stream
// serialisation the next step's CTAs take the slots this step's CTAs free and wait
// on the device for its completion, so consecutive steps' launch latency and CTA ramp
// overlap the previous step's tail.  The row kernels, single and batch, one CTA per SM,
// always are (lbm_row.cu); so are the persistent tile kernels when their CTAs take
// several work items in turn (256^3: 499 -> 488 us).  A grid of one item per CTA has no
// such tail and measured 0.6 us slower with it (128^3), the tile kernels' batches 26%
// slower over a 144-lattice sweep, and the two passes much slower (32^3 FP64 13.6 -> 47 us:
// waiting CTAs crowd the SMs that free first): these are launched plainly.
template <typename... KArgs, typename... Args>
static cudaError_t launch_step_kernel(void (*kern)(KArgs...), long long grid, int threads, size_t smem,
                                      cudaStream_t s, bool overlap, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = overlap ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

}  // namespace lbm
