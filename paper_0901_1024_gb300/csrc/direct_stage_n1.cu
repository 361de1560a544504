// One-thread-per-element stage, order 1.
#include "direct_stage.cuh"

namespace dgdev {

cudaError_t launch_direct_stage(bool rk, const StageArgs& a, const DirectOps<1>& o, cudaStream_t s) {
  const bool ext = a.mat || a.absorbing;
  auto kern = rk ? (ext ? direct_stage_kernel<1, true, true> : direct_stage_kernel<1, true, false>)
                 : (ext ? direct_stage_kernel<1, false, true> : direct_stage_kernel<1, false, false>);
  if (a.num_tiles <= 0) return cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((a.num_tiles + kDirectThreads - 1) / kDirectThreads);
  cfg.blockDim = dim3(kDirectThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a, o);
}

}  // namespace dgdev
