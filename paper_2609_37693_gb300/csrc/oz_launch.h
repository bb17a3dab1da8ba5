// oz_launch.h -- kernel launches with programmatic stream serialisation: the
// kernel may be scheduled while its predecessor on the stream drains, so the
// launch latency and the set-up of one phase run under the tail of the phase
// before. Only a kernel that calls pdl_wait (oz_device.cuh) before it touches
// global memory may be launched dependent: the joint splits (split_both_kernel,
// split_tiles_kernel), the GEMMs of one product (gemm_tc_kernel,
// gemm_tc_pair_kernel) and reconstruct_groups8_kernel. All others have no wait
// and are correct in plain stream order only.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace oz {

// Outputs from this many entries on are launched in plain stream order. A
// dependent launch is worth 2 us at 2048^3 (285 against 287) and most of the
// gaps of a small product, but cost a larger one more than that: 2400 x 2400 x
// 512 200 us against 191, 3000 x 2500 x 2000 507 against 499, 65536 x 256 x 256
// 390 us against 382, 8192 x 8192 x 256 1001 against 978, 16384^3 94.9 ms
// against 94.3.
constexpr int64_t kDependentMaxOutput = 5ll << 20;

// Whether the GEMM and the reconstruct of an m x n output are launched dependent.
inline bool dependent_suits(int64_t m, int64_t n) { return n == 0 || m < kDependentMaxOutput / n; }

// cluster: blocks per cluster (1 also for kernels with __cluster_dims__)
template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel(bool dependent, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                                 cudaStream_t st, int cluster, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2] = {};
  if (dependent) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster > 1) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    attr[cfg.numAttrs].val.clusterDim.x = (unsigned)cluster;
    attr[cfg.numAttrs].val.clusterDim.y = attr[cfg.numAttrs].val.clusterDim.z = 1;
    ++cfg.numAttrs;
  }
  cfg.attrs = attr;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

}  // namespace oz
