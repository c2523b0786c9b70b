// Instantiations of the fused kernels for scenes that hold mesh objects (the
// lookup dispatches on the object kind); grid-only scenes use the kernels of
// fg_fused.cu / fg_fused_opt.cu, which compile the grid lookup alone.
#include "fg_fused_kernel.cuh"

namespace fg {

#define FG_CFG_LOSSGRAD_ANY(nw, mb, ppt) &launch_fused_cfg<kModeLossGrad, nw, mb, ppt, true>,
extern const FusedLaunchFn kLossGradLaunchAny[] = {FG_FUSED_CONFIGS(FG_CFG_LOSSGRAD_ANY)};

// Scenes with grids whose gradient is zero in cells that can be in contact: one configuration a
// mode, whatever is selected.
cudaError_t launch_fused_flat(int mode, const FusedArgs& a, cudaStream_t st) {
  switch (mode) {
    case kModeWrench: return launch_fused_cfg<kModeWrench, 4, 5, 1, true, true>(a, st);
    case kModeLossGrad: return launch_fused_cfg<kModeLossGrad, 8, 3, 1, true, true>(a, st);
    case kModeQueue: return launch_fused_cfg<kModeQueue, 4, 5, 1, true, true>(a, st);
    default: return launch_fused_cfg<kModeOptimize, 8, 3, 1, true, true>(a, st);
  }
}

cudaError_t launch_wrench_any(const FusedArgs& a, cudaStream_t st) {
  return launch_fused_cfg<kModeWrench, 4, 5, 1, true>(a, st);
}

cudaError_t launch_queue_round_any(const FusedArgs& a, cudaStream_t st) {
  return launch_fused_cfg<kModeQueue, 4, 5, 1, true>(a, st);
}

}  // namespace fg
