// One-thread-per-element stage, order 1.
#include "direct_stage.cuh"

namespace dgdev {

template <bool RK>
static auto direct_kernel(Ext ext) {
  switch (ext) {
    case Ext::absorbing: return direct_stage_kernel<1, RK, Ext::absorbing>;
    case Ext::materials: return direct_stage_kernel<1, RK, Ext::materials>;
    case Ext::any: return direct_stage_kernel<1, RK, Ext::any>;
    default: return direct_stage_kernel<1, RK, Ext::none>;
  }
}

cudaError_t launch_direct_stage(bool rk, const StageArgs& a, const DirectOps<1>& o, int num_sms,
                                cudaStream_t s) {
  if (a.num_tiles <= 0) return cudaSuccess;
  const int grid = (a.num_tiles + kDirectThreads - 1) / kDirectThreads;
  auto kern = rk ? direct_kernel<true>(direct_ext(a.mat, a.absorbing, grid, num_sms))
                 : direct_kernel<false>(direct_ext(a.mat, a.absorbing, grid, num_sms));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
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
