// The T-step kernel for scenes with grids whose gradient is zero in cells that can be in contact
// (FusedArgs::any_flat), 8 warps a candidate; apart from fg_tstep.cu so that they compile in parallel.
#include "fg_tstep_kernel.cuh"

namespace fg {

template <bool ANY>
static cudaError_t launch_flat(int mode, const FusedArgs& a, cudaStream_t st) {
  return mode == kModeLossGrad ? launch_tstep_mode<kModeLossGrad, ANY, kTWide, true>(a, st)
                               : launch_tstep_mode<kModeOptimize, ANY, kTWide, true>(a, st);
}

cudaError_t launch_tstep_flat(int mode, const FusedArgs& a, cudaStream_t st) {
  return a.any_mesh ? launch_flat<true>(mode, a, st) : launch_flat<false>(mode, a, st);
}

}  // namespace fg
