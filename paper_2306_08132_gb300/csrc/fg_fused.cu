// Dispatch of the fused kernels: compiled configurations, the per-device
// selection, and the autotuner that times the configurations on a workload.
#include <cuda_runtime.h>

#include "fg_fused_kernel.cuh"

namespace fg {

#define FG_CFG_NW(nw, mb, ppt) nw,
#define FG_CFG_MB(nw, mb, ppt) mb,
#define FG_CFG_PPT(nw, mb, ppt) ppt,
#define FG_CFG_LOSSGRAD(nw, mb, ppt) &launch_fused_cfg<kModeLossGrad, nw, mb, ppt>,
static const int kCfgNW[] = {FG_FUSED_CONFIGS(FG_CFG_NW)};
static const int kCfgMinB[] = {FG_FUSED_CONFIGS(FG_CFG_MB)};
static const int kCfgPPT[] = {FG_FUSED_CONFIGS(FG_CFG_PPT)};
static const FusedLaunchFn kLossGradLaunch[] = {FG_FUSED_CONFIGS(FG_CFG_LOSSGRAD)};
constexpr int kNumCfg = sizeof(kCfgNW) / sizeof(kCfgNW[0]);
constexpr int kCfg4 = 1;         // 4 warps per candidate, >= 5 CTAs per SM, 1 point per thread
constexpr int kCfg8 = 4;         // 8 warps, >= 3 CTAs per SM
constexpr int kCfg16 = 11;       // 16 warps, >= 1 CTA per SM

// Warps per candidate of a launch without a selected configuration.  With few
// candidates the chip is filled by giving each more warps (ms with 4, 8, 16 warps;
// 4,352 points): 152 candidates 0.100, 0.069, 0.049; 456: 0.145, 0.102, 0.099; 912: 0.189,
// 0.150, 0.166; 1,824: 0.251, 0.225, 0.297; 4,096: 0.433, 0.445, 0.626.  A small hand has too
// few chunks to share (640 points: 152 candidates 0.041, 0.033, 0.028; 304: 0.044, 0.037,
// 0.044; 912: 0.058, 0.059, 0.092).  On a mesh a candidate inside the object costs many
// times the others, so more warps shorten the end of the launch (4,352 points, 2,208 faces: 1,024
// candidates 2.11, 1.40, 1.29; 4,096: 6.03, 4.49, 4.08; 8,192: 9.55, 7.15, 7.34; other hands on
// meshes were not measured).
// The configuration changes no result: units, chunks and sums are the same at any number of warps.
static int default_config(const FusedArgs& a) {
  const long long sms = device_sm_count(), B = a.B;
  const bool large = a.hand_P >= 2048;
  if (a.any_mesh) return B <= 32 * sms ? kCfg16 : kCfg8;
  if (B <= (large ? 3 : 1) * sms) return kCfg16;
  return B <= (large ? 12 : 4) * sms ? kCfg8 : kCfg4;
}

static int g_selected[64] = {-1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1,
                             -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1,
                             -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1,
                             -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1};

int fused_config_count() { return kNumCfg; }
void fused_config_info(int i, int* nw, int* minb, int* ppt) {
  *nw = kCfgNW[i];
  *minb = kCfgMinB[i];
  *ppt = kCfgPPT[i];
}
static int& selected_slot() {
  int dev = 0;
  cudaGetDevice(&dev);
  return g_selected[dev & 63];
}
// -1 when none is selected (each launch then follows default_config).
int fused_config_current() { return selected_slot(); }
void fused_config_select(int i) { selected_slot() = i; }

cudaError_t launch_fused(int mode, const FusedArgs& a, const fg_hand* h, cudaStream_t st) {
  (void)h;
  if (a.B <= 0) return cudaSuccess;
  const int chosen = selected_slot(), cfg = chosen < 0 ? default_config(a) : chosen;
  if (a.any_flat) return launch_fused_flat(mode, kCfgNW[cfg] > 4, a, st);
  if (a.any_mesh) {
    switch (mode) {
      case kModeWrench: return launch_wrench_any(a, st);
      case kModeLossGrad: return kLossGradLaunchAny[cfg](a, st);
      default: return kOptimizeLaunchAny[cfg](a, st);
    }
  }
  switch (mode) {
    case kModeWrench: return launch_fused_cfg<kModeWrench, 4, 5, 1>(a, st);
    case kModeLossGrad: return kLossGradLaunch[cfg](a, st);
    default: return kOptimizeLaunch[cfg](a, st);
  }
}

// One round of a request queue: every active request's candidates in one launch.
cudaError_t launch_queue_round(const FusedArgs& a, cudaStream_t st) {
  if (a.B <= 0) return cudaSuccess;
  if (a.any_flat) return launch_fused_flat(kModeQueue, false, a, st);
  if (a.any_mesh) return launch_queue_round_any(a, st);
  return launch_fused_cfg<kModeQueue, 4, 5, 1>(a, st);
}

cudaError_t autotune_fused(const FusedArgs& base, int reps, float* times_ms, int* best, cudaStream_t st) {
  const size_t qbytes = sizeof(float) * (size_t)base.B * 64;
  (void)qbytes;
  float* qtmp = nullptr;
  float* ltmp = nullptr;
  const int D = base.hand_D;
  cudaError_t e = cudaMallocAsync(&qtmp, sizeof(float) * (size_t)base.B * D, st);
  if (e != cudaSuccess) return e;
  e = cudaMallocAsync(&ltmp, sizeof(float) * (size_t)base.B, st);
  if (e != cudaSuccess) {
    cudaFreeAsync(qtmp, st);
    return e;
  }
  cudaEvent_t t0, t1;
  cudaEventCreate(&t0);
  cudaEventCreate(&t1);
  float best_ms = 3.0e38f;
  int best_i = kCfg4;
  for (int i = 0; i < kNumCfg && e == cudaSuccess; ++i) {
    FusedArgs a = base;
    a.q = qtmp;
    a.loss = ltmp;
    float total = 0.0f;
    for (int r = 0; r <= reps && e == cudaSuccess; ++r) {   // r = 0 warms up
      e = cudaMemcpyAsync(qtmp, base.q, sizeof(float) * (size_t)base.B * D, cudaMemcpyDeviceToDevice, st);
      if (e != cudaSuccess) break;
      cudaEventRecord(t0, st);
      e = base.any_flat ? launch_fused_flat(kModeOptimize, kCfgNW[i] > 4, a, st)
                        : (base.any_mesh ? kOptimizeLaunchAny : kOptimizeLaunch)[i](a, st);
      cudaEventRecord(t1, st);
      if (e == cudaSuccess) e = cudaEventSynchronize(t1);
      float ms = 0.0f;
      cudaEventElapsedTime(&ms, t0, t1);
      if (r > 0) total += ms;
    }
    const float avg = total / (reps > 0 ? reps : 1);
    if (times_ms) times_ms[i] = avg;
    if (avg < best_ms) {
      best_ms = avg;
      best_i = i;
    }
  }
  cudaEventDestroy(t0);
  cudaEventDestroy(t1);
  cudaFreeAsync(qtmp, st);
  cudaFreeAsync(ltmp, st);
  if (e == cudaSuccess) {
    fused_config_select(best_i);
    if (best) *best = best_i;
  }
  return e;
}

}  // namespace fg
