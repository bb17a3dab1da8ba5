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

// Outputs from this many entries on are launched in plain stream order. What
// a dependent launch costs them is the reconstruct's L1: its blocks start on SMs
// that still hold a GEMM block, so they keep that block's split of the SM's memory,
// nearly all of it shared, where a plain launch gives L1 the larger part. At
// 2400^2 the reconstruct takes 61.7 us, and 78.1 launched plain with all memory asked
// for as shared; at 4096^2 99 and 114. The gaps that the two dependent launches hide
// are worth a few microseconds whatever the size, so the line lies where the two
// together stop gaining, between 4 Mi entries (1.5 us gained) and 5.8 Mi (12 lost).
// Products, us, both plain / GEMM dependent / reconstruct dependent / both:
//   1024 x 1024 x 1024   78.4   75.9   73.9   70.7
//   2048 x 2048 x 2048    285    282    286    283
//   2400 x 2400 x 512     184    182    198    196
//   3000 x 2500 x 2000    491    487    506    503
//   65536 x 256 x 256     371    368    381    379
//   8192 x 8192 x 256     934    931    982    977
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
