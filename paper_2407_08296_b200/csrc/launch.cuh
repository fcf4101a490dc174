// Kernel launches that may overlap the launch before them in the stream (programmatic stream serialization).
#pragma once

#include <cuda_runtime.h>

#include <utility>

#include "qg_common.cuh"

namespace qg {

// The grid may begin while the launch before it drains: its CTAs are scheduled, and run up to their grid_dependency_wait,
// once every CTA of that launch has called grid_launch_dependents or left.  The kernel has to call grid_dependency_wait
// before it touches anything an earlier launch may write or read; a launch before it that knows nothing of this (another
// library's kernel, a copy) is simply waited for.  `cluster`: CTAs per cluster.
template <class... Params, class... Args>
int launch_overlapping(void (*kern)(Params...), unsigned grid, unsigned block, size_t smem, cudaStream_t st, unsigned cluster, Args&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2]{};
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  QG_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...));
  count_launch();
  return QG_OK;
}

}  // namespace qg
