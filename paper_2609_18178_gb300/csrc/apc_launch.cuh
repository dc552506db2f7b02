// The launches of a call whose table takes several.  Where the grid may take the
// whole GPU they are chained: each but the last lets the next start at once
// (griddepcontrol.launch_dependents), and each but the first is launched with
// programmatic stream serialization, so it may: its CTAs move onto the SMs as
// the ones before leave them, where an ordinary launch would begin after the
// last CTA of the one before, with a gap of its own.  The launches touch
// disjoint ranges; only their sums meet in the output, and each waits
// (griddepcontrol.wait) before it adds its own until the one before has
// completed, so the last one completes last.  It lets nothing start early:
// whatever follows on the stream waits for it as for any kernel.  Where SMs are
// to stay free the launches are ordinary ones: a chained launch's CTAs would
// take those SMs and sit there until the launch before has ended.
//
// Measured against ordinary launches: 4,400 buffers in five launches verify in
// 104 us (119) with the wait for them, 69 (75) among other calls; 1,100 tensors
// in three launches commit in 120 us (133) and 83 (86).  The
// output's zeroing stays a memset: a zeroing kernel that let a single working
// kernel start early took 1.6 us off a 22 us call but added 0.5 to 2 us of host
// time to every call.
#pragma once

#include <cuda_runtime.h>

namespace apc {

// chained: not the first launch of its call.
template <class Plan>
int launch_plan(void (*kernel)(Plan, unsigned long long *), const Plan &plan, bool chained, unsigned grid,
                unsigned threads, unsigned smem, void *stream, unsigned long long *out) {
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = (cudaStream_t)stream;
  cfg.attrs = &attr;
  cfg.numAttrs = chained ? 1 : 0;
  return (int)cudaLaunchKernelEx(&cfg, kernel, plan, out);
}

}  // namespace apc
