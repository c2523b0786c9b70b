// Launch of the T-step kernel (fg_tstep_kernel.cuh).
#include "fg_tstep_kernel.cuh"

namespace fg {

namespace {

template <int TW>
cudaError_t launch_tstep_warps(int mode, const FusedArgs& a, cudaStream_t st) {
  if (a.any_mesh)
    return mode == kModeLossGrad ? launch_tstep_mode<kModeLossGrad, true, TW>(a, st)
                                 : launch_tstep_mode<kModeOptimize, true, TW>(a, st);
  return mode == kModeLossGrad ? launch_tstep_mode<kModeLossGrad, false, TW>(a, st)
                               : launch_tstep_mode<kModeOptimize, false, TW>(a, st);
}

}  // namespace

cudaError_t launch_tstep(int mode, const FusedArgs& a, cudaStream_t st) {
  if (a.B <= 0) return cudaSuccess;
  if (a.P.sim_steps < 1 || a.P.sim_steps > kTSteps) return cudaErrorInvalidValue;
  if (a.any_flat) return launch_tstep_flat(mode, a, st);
  // Eight warps a candidate shorten its phases and fill the chip with few candidates (4,352
  // points, T = 1: 152 candidates 0.217 -> 0.136 ms, 912: 0.444 -> 0.364, 2,048: 0.693 -> 0.663,
  // 4,096: 1.197 -> 1.235; 640 points: 304 candidates 0.082 -> 0.065, 608: 0.085 -> 0.092), and the sweeps
  // of the later steps balance better over them at any number (T = 2: 152 candidates 0.589 -> 0.354,
  // 4,096: 4.18 -> 3.89; 640 points, 4,096: 1.25 -> 1.13).
  const bool wide = a.P.sim_steps >= 2 || a.B <= (a.hand_P >= 2048 ? 12LL : 3LL) * device_sm_count();
  return wide ? launch_tstep_warps<kTWide>(mode, a, st) : launch_tstep_warps<kTWarps>(mode, a, st);
}

}  // namespace fg
