// Kernel launches that may overlap the launch before them in the stream (programmatic stream serialization).
#pragma once

#include <cuda_runtime.h>

#include <utility>

#include "qg_common.cuh"

namespace qg {

// The grid may begin while the launch before it drains: its CTAs are scheduled, and run up to their grid_dependency_wait,
// once every CTA of that launch has called grid_launch_dependents or left.  The kernel has to call grid_dependency_wait
// before it touches anything an earlier launch may write or read; a launch before it that knows nothing of this (another
// library's kernel, a copy) is simply waited for.  `cluster`: CTAs per cluster; `overlap` = false: an ordinary launch.
//
// What keeps this sound:
//  - A kernel calls grid_launch_dependents only after its own grid_dependency_wait (or in an ordinary launch), so a launch begins
//    when the one before the one before it is complete: two are in flight at most, and what a kernel reads through the read-only
//    path (scales that an earlier step wrote, a new projection) was written by CTAs that had left before this launch began.
//  - It calls it only when its CTA has its tensor memory.  tcgen05.alloc waits without a limit: a CTA of the later launch that took
//    an SM's columns first, and then waited for the earlier launch, would never give them back.  No two CTAs that allocate tensor
//    memory fit an SM together either: each such kernel takes more than half of its shared memory.
constexpr int kHalfOfSharedMemory = 228 * 1024 / 2;

template <class... Params, class... Args>
int launch_overlapping(void (*kern)(Params...), unsigned grid, unsigned block, size_t smem, cudaStream_t st, unsigned cluster, bool overlap,
                       Args&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2]{};
  if (overlap) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster > 1) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    attr[cfg.numAttrs].val.clusterDim.x = cluster;
    attr[cfg.numAttrs].val.clusterDim.y = 1;
    attr[cfg.numAttrs++].val.clusterDim.z = 1;
  }
  cfg.attrs = attr;
  QG_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...));
  count_launch();
  return QG_OK;
}

}  // namespace qg
