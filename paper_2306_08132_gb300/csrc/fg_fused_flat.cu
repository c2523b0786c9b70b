// Instantiations of the fused kernels for scenes with grids whose gradient is zero in cells that
// can be in contact (FusedArgs::any_flat): two further passes add those contacts' friction and its
// adjoint.  One configuration of 4 and one of 8 warps for grids, one of 8 with mesh objects.
#include "fg_fused_kernel.cuh"

namespace fg {

template <int MODE>
static cudaError_t launch_flat_step(bool wide, const FusedArgs& a, cudaStream_t st) {
  if (a.any_mesh) return launch_fused_cfg<MODE, 8, 3, 1, true, true>(a, st);
  return wide ? launch_fused_cfg<MODE, 8, 3, 1, false, true>(a, st) : launch_fused_cfg<MODE, 4, 5, 1, false, true>(a, st);
}

template <int MODE>
static cudaError_t launch_flat_four(const FusedArgs& a, cudaStream_t st) {
  return a.any_mesh ? launch_fused_cfg<MODE, 4, 5, 1, true, true>(a, st) : launch_fused_cfg<MODE, 4, 5, 1, false, true>(a, st);
}

// wide: more than 4 warps a candidate (loss and gradient, optimisation steps).
cudaError_t launch_fused_flat(int mode, bool wide, const FusedArgs& a, cudaStream_t st) {
  switch (mode) {
    case kModeWrench: return launch_flat_four<kModeWrench>(a, st);
    case kModeQueue: return launch_flat_four<kModeQueue>(a, st);
    case kModeLossGrad: return launch_flat_step<kModeLossGrad>(wide, a, st);
    default: return launch_flat_step<kModeOptimize>(wide, a, st);
  }
}

}  // namespace fg
