// Grasp-quality metrics of the paper's evaluation (Sec. V, "Metrics") for batches
// of candidates: the weighted contact measure (contact area CA with surface
// samples and area weights, intersection volume IV with interior samples and
// volume weights) and epsilon over a set of wrench-space directions.
//
// Contacts are the hand points with phi(p) < tau (undilated SDF, object at its
// canonical pose).  A contact with outward normal n contributes the k edges of
// its Coulomb cone, f_e = -n + mu (cos(2 pi e/k) t1 + sin(2 pi e/k) t2) with the
// tangent basis (t1, t2) of Duff et al. (2017), as wrenches
// w = (f, s (p - c) x f), s the torque scale and c the object's origin.  For a
// unit direction u = (u_f, u_t), u . w = a . f with a = u_f + s (u_t x p), so
//   max_e u . w_e = -a . n + mu max_e (cos_e a . t1 + sin_e a . t2),
// and eps_U = min over the directions of the maximum over all contacts.
//
// Both kernels: one CTA per candidate (persistent, candidates claimed from a
// counter), FK by warp 0; a chunk of 32 points whose bounding sphere has
// sphere_bound >= tau holds no contact and is left out (a quarter of the chunks stays
// at tau = 5 mm), and a chunk that stays is tested point by point on the min-pyramid
// before its lookups.  Epsilon collects the contacts of 32 chunks at a time in
// shared memory (point, normal, tangent basis); the threads fold them into the
// running maxima of the directions; max and min do not depend on order, so the
// result is exact with respect to the order of the contacts.
#include <cuda_runtime.h>

#include <math.h>

#include "fg_fused_kernel.cuh"
#include "fg_internal.h"

namespace fg {

namespace {

constexpr int kQW = 8;                       // warps per candidate
constexpr int kQBatchChunks = 32;            // chunks per contact batch (<= 1024 contacts)
constexpr int kQBatch = 32 * kQBatchChunks;
constexpr int kQD = 2;                       // directions per thread per pass over the contacts

struct QualitySmem {
  HandDev H;
  float4 frame4[kMaxLinks][3];
  float q[64];
  float red[kQW];
  float ce[32], se[32];                      // cone edge angles
  int count;
  int total;
  unsigned bits[kMaxCullChunks / 32];        // chunks that may hold a contact
  ObjDev O;
  int bad_object;
  int cand;                                  // the candidate claimed by this CTA
  const HandDev* hand_loaded;
};

// Loads the hand descriptor (if it changed) and the candidate's object and q,
// then computes the link frames.  Returns false for an object index outside the scene.
__device__ bool quality_setup(QualitySmem& S, const FusedArgs& a, int c, int tid, int nthreads) {
  __syncthreads();
  if (tid == 0) {
    const int oi = a.obj_of_cand ? a.obj_of_cand[c] : 0;
    S.bad_object = oi < 0 || oi >= a.n_obj;
    if (!S.bad_object) S.O = a.objs[oi];
  }
  if (a.hand != S.hand_loaded) {
    const int* src = reinterpret_cast<const int*>(a.hand);
    int* dst = reinterpret_cast<int*>(&S.H);
    for (int k = tid; k < (int)(sizeof(HandDev) / sizeof(int)); k += nthreads) dst[k] = src[k];
  }
  __syncthreads();
  if (tid == 0) S.hand_loaded = a.hand;
  if (tid < S.H.D) S.q[tid] = a.q[(size_t)c * S.H.D + tid];
  __syncthreads();
  if (S.bad_object) return false;
  if (tid < 32) fk_warp(S.H, S.q, S.frame4, tid);
  __syncthreads();
  return true;
}

// Marks the chunks that may hold a point with phi < tau in S.bits.  Hands with more
// chunks than S.bits holds keep all of them.
template <bool ANY>
__device__ __forceinline__ void quality_cull(QualitySmem& S, float tau, int lane, int warp) {
  const HandDev& H = S.H;
  if (H.nchunks <= kMaxCullChunks) {
    for (int j0 = 32 * warp; j0 < H.nchunks; j0 += 32 * kQW) {
      const int j = j0 + lane;
      bool keep = j < H.nchunks;
      if (keep) {
        const int l = H.chunk_link[j];
        keep = l < 0 || !(sphere_bound<ANY>(S.O, S.frame4[l], __ldg(H.chunk_sphere + j)) - tau > 0.0f);
      }
      const unsigned word = __ballot_sync(kFull, keep);
      if (lane == 0) S.bits[j0 >> 5] = word;
    }
  }
  __syncthreads();
}
__device__ __forceinline__ bool quality_culled(const QualitySmem& S, int j) {
  return S.H.nchunks <= kMaxCullChunks && !((S.bits[j >> 5] >> (j & 31)) & 1u);
}

// Lookup of lane's point of chunk j: true when it is a contact (phi < tau).  A chunk
// none of whose points can be one (a pyramid entry each) skips the lookups.
template <bool ANY>
__device__ __forceinline__ bool quality_lookup(const QualitySmem& S, int j, int lane, float tau, float p[3],
                                               SdfSample& smp) {
  const HandDev& H = S.H;
  const int i = 32 * j + lane;
  const bool valid = i < H.P;
  const float4 sp = __ldg(H.pts + (valid ? i : 32 * j));
  world_point(S.frame4[(int)sp.w], sp, p);
  if (!(ANY && S.O.kind == kObjMesh)) {
    const float mn = point_min_bound(S.O, p);
    if (__all_sync(kFull, !valid || mn - tau - (1e-6f + 1e-5f * fabsf(mn)) > 0.0f)) return false;
  }
  sdf_lookup<false, ANY>(S.O, p, smp);
  return valid && smp.phi < tau;
}

// Bound: the culling's 27 pyramid reads a chunk and the lookups of the chunks that
// stay, both latency; 8,192 candidates of 4,352 points at 5 mm:
// 0.45 -> 0.13 ms, L1 data pipe 48%, FK by one warp leaves the others at the barrier.
template <bool ANY>
__global__ void __launch_bounds__(kQW * 32) measure_kernel(FusedArgs a, const float* __restrict__ weights, float tau,
                                                        float* __restrict__ out) {
  __shared__ QualitySmem S;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) S.hand_loaded = nullptr;
  for (;;) {
    const int c = next_candidate(a.work, &S.cand);
    if (c >= a.B) break;
    if (!quality_setup(S, a, c, tid, kQW * 32)) {
      if (tid == 0) out[c] = __int_as_float(0x7fc00000);
      continue;
    }
    quality_cull<ANY>(S, tau, lane, warp);
    const HandDev& H = S.H;
    float acc = 0.0f;
    for (int j = warp; j < H.nchunks; j += kQW) {      // chunk j to warp j mod 8: a fixed order of additions
      if (quality_culled(S, j)) continue;
      float p[3];
      SdfSample smp;
      if (quality_lookup<ANY>(S, j, lane, tau, p, smp)) acc += __ldg(weights + 32 * j + lane);
    }
    acc = warp_sum(acc);
    if (lane == 0) S.red[warp] = acc;
    __syncthreads();
    if (tid == 0) {
      float t = 0.0f;
#pragma unroll
      for (int w = 0; w < kQW; ++w) t += S.red[w];
      out[c] = t;
    }
  }
  work_done(a.work);
}

// Two contacts of the batch, value by value (x: the even one, y: the odd one): point p,
// outward normal n, tangent basis t1, t2.
struct ContactPair {
  float2 p[3], n[3], t1[3], t2[3];
};

// max over the k cone edges of cos_e x + sin_e y, from the edges that can attain it.
// The edges are symmetric under y -> -y, for even k under x -> -x and for k a
// multiple of 4 under x <-> y, so after the matching reflections the angle of (x, y)
// lies in [0, pi], [0, pi/2] or [0, pi/4] and only edges 0 .. last = k/2, k/4 or k/8 (rounded down)
// can be the nearest.  Edge 0 is (1, 0).  EIGHT (k = 8) needs no order of |x| and |y|:
// max(|x|, |y|, (|x| + |y|)/sqrt 2), 3 operations instead of 24.
enum ConeSymmetry { kConeOdd = 0, kConeEven = 1, kConeQuad = 2 };
__device__ __forceinline__ int cone_symmetry(int k) { return (k & 1) ? kConeOdd : (k & 3) ? kConeEven : kConeQuad; }
__device__ __forceinline__ int cone_last_edge(int k) { return (k & 1) ? k / 2 : (k & 3) ? k / 4 : k / 8; }

template <bool EIGHT>
__device__ __forceinline__ float cone_max(float a1, float a2, const float* ce, const float* se, int sym, int last) {
  if (EIGHT) return fmaxf(fmaxf(fabsf(a1), fabsf(a2)), ce[1] * (fabsf(a1) + fabsf(a2)));
  float y = fabsf(a2), x = sym == kConeOdd ? a1 : fabsf(a1);
  if (sym == kConeQuad) {
    const float t = fmaxf(x, y);
    y = fminf(x, y);
    x = t;
  }
  float best = x;
  for (int e = 1; e <= last; ++e) best = fmaxf(best, ce[e] * x + se[e] * y);
  return best;
}

// Running maxima h of kQD directions over the contact pairs j0, j0 + stride, ...: the dot
// products of both contacts of a pair in packed f32x2 arithmetic, every value of a
// direction twice in a register pair.
template <bool EIGHT>
__device__ __forceinline__ void fold_contacts(const ContactPair* rec, int np, int j0, int stride, const float* ce,
                                              const float* se, int sym, int last, float mu,
                                              const float (&uf)[kQD][3], const float (&ut)[kQD][3], float (&h)[kQD]) {
  float2 f2[kQD][3], t2[kQD][3], m2[kQD][3];
#pragma unroll
  for (int d = 0; d < kQD; ++d)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      f2[d][k] = make_float2(uf[d][k], uf[d][k]);
      t2[d][k] = make_float2(ut[d][k], ut[d][k]);
      m2[d][k] = make_float2(-ut[d][k], -ut[d][k]);
    }
  for (int jp = j0; jp < np; jp += stride) {
    const ContactPair c = rec[jp];
#pragma unroll
    for (int d = 0; d < kQD; ++d) {
      // a = u_f + s (u_t x p)
      const float2 a[3] = {vfma(m2[d][2], c.p[1], vfma(t2[d][1], c.p[2], f2[d][0])),
                           vfma(m2[d][0], c.p[2], vfma(t2[d][2], c.p[0], f2[d][1])),
                           vfma(m2[d][1], c.p[0], vfma(t2[d][0], c.p[1], f2[d][2]))};
      const float2 an = vdot(a, c.n), a1 = vdot(a, c.t1), a2 = vdot(a, c.t2);
      const float vx = mu * cone_max<EIGHT>(a1.x, a2.x, ce, se, sym, last) - an.x;
      const float vy = mu * cone_max<EIGHT>(a1.y, a2.y, ce, se, sym, last) - an.y;
      h[d] = fmaxf(h[d], fmaxf(vx, vy));
    }
  }
}

// Floats as integers of the same order, for atomicMax in shared memory (no NaN arrives here).
__device__ __forceinline__ int float_order(float x) {
  const int i = __float_as_int(x);
  return i >= 0 ? i : i ^ 0x7fffffff;
}
__device__ __forceinline__ float order_float(int i) { return __int_as_float(i >= 0 ? i : i ^ 0x7fffffff); }

// Bound: issue in the fold, 13 instructions a (direction, contact) pair with 8 edges.
// 8,192 candidates, 76 contacts each, 1,024 directions, 8 edges: 2.27 -> 0.77 to 0.80 ms (FMA
// pipe 33%; the SMs are busy 73% of the launch: candidates with over a
// thousand contacts end last).
template <bool ANY>
__global__ void __launch_bounds__(kQW * 32) epsilon_kernel(FusedArgs a, float tau, float mu, int k_edges,
                                                        float tscale, const float* __restrict__ dirs, int K,
                                                        float* __restrict__ eps, int* __restrict__ ncontact) {
  __shared__ QualitySmem S;
  __shared__ unsigned short list[kQBatchChunks];
  extern __shared__ float4 dyn4[];
  ContactPair* rec = reinterpret_cast<ContactPair*>(dyn4);      // [kQBatch / 2]
  int* hmax = reinterpret_cast<int*>(rec + kQBatch / 2);        // [K], float_order
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int NT = kQW * 32;
  if (tid == 0) S.hand_loaded = nullptr;
  if (tid < 32) {
    float s, co;
    sincospif(2.0f * (float)tid / (float)k_edges, &s, &co);
    S.ce[tid] = co;
    S.se[tid] = s;
  }
  const int sym = cone_symmetry(k_edges), last = cone_last_edge(k_edges);
  // Each thread takes kQD directions; with fewer than NT * kQD of them the contacts
  // are dealt out to `ways` groups of threads.
  const int groups = (K + kQD - 1) / kQD;
  const int ways = groups < NT ? NT / groups : 1;
  for (;;) {
    const int c = next_candidate(a.work, &S.cand);
    if (c >= a.B) break;
    if (!quality_setup(S, a, c, tid, NT)) {
      if (tid == 0) {
        eps[c] = __int_as_float(0x7fc00000);
        if (ncontact) ncontact[c] = -1;
      }
      continue;
    }
    const HandDev& H = S.H;
    for (int k = tid; k < K; k += NT) hmax[k] = float_order(-INFINITY);
    if (tid == 0) S.total = 0;
    quality_cull<ANY>(S, tau, lane, warp);
    int next = 0;                                       // first chunk not yet listed
    while (next < H.nchunks) {
      // the next kQBatchChunks chunks that may hold a contact (every warp finds the
      // same ones; warp 0 lists them)
      int n = 0;
      while (n < kQBatchChunks && next < H.nchunks) {
        const int j = next + lane;
        const unsigned open_ = __ballot_sync(kFull, j < H.nchunks && !quality_culled(S, j));
        const int rank = n + __popc(open_ & ((1u << lane) - 1u));
        const bool mine = (open_ >> lane) & 1u;
        if (warp == 0 && mine && rank < kQBatchChunks) list[rank] = (unsigned short)j;
        const unsigned over = __ballot_sync(kFull, mine && rank >= kQBatchChunks);
        n = min(n + __popc(open_), kQBatchChunks);
        next += over ? __ffs(over) - 1 : 32;
      }
      if (n == 0) break;
      if (tid == 0) S.count = 0;
      __syncthreads();
      for (int idx = warp; idx < n; idx += kQW) {
        const int j = list[idx];
        float p[3];
        SdfSample smp;
        const bool hit = quality_lookup<ANY>(S, j, lane, tau, p, smp);
        const unsigned bal = __ballot_sync(kFull, hit);
        int base = 0;
        if (lane == 0 && bal) base = atomicAdd(&S.count, __popc(bal));
        base = __shfl_sync(kFull, base, 0);
        if (hit) {
          const float g2 = smp.g[0] * smp.g[0] + smp.g[1] * smp.g[1] + smp.g[2] * smp.g[2];
          const float rg = rsqrt_or_zero(g2);
          const float nr[3] = {smp.g[0] * rg, smp.g[1] * rg, smp.g[2] * rg};
          // Duff et al. (2017): s = sign(n_z) (+1 at 0), a = -1/(s + n_z), b = n_x n_y a
          const float sg = nr[2] >= 0.0f ? 1.0f : -1.0f;
          const float aa = -1.0f / (sg + nr[2]);
          const float bb = nr[0] * nr[1] * aa;
          const float t1[3] = {1.0f + sg * nr[0] * nr[0] * aa, sg * bb, -sg * nr[0]};
          const float t2[3] = {bb, sg + nr[1] * nr[1] * aa, -nr[1]};
          const int slot = base + __popc(bal & ((1u << lane) - 1u));
          float* w = reinterpret_cast<float*>(rec + (slot >> 1)) + (slot & 1);
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            w[2 * k] = p[k];
            w[2 * (3 + k)] = nr[k];
            w[2 * (6 + k)] = t1[k];
            w[2 * (9 + k)] = t2[k];
          }
        }
      }
      __syncthreads();
      const int nc = S.count, np = (nc + 1) >> 1;
      if (nc & 1) {                                     // the last contact stands twice
        if (tid < 12) {
          float* w = reinterpret_cast<float*>(rec + np - 1) + 2 * tid;
          w[1] = w[0];
        }
        __syncthreads();
      }
      // kQD directions per thread per pass: each contact record read from shared
      // memory serves all of them
      for (int w0 = tid; w0 < groups * ways && nc > 0; w0 += NT) {
        const int way = w0 / groups, k0 = w0 - way * groups;       // directions k0, k0 + groups, ...
        float uf[kQD][3], ut[kQD][3], h[kQD];
#pragma unroll
        for (int d = 0; d < kQD; ++d) {
          const int k = min(k0 + d * groups, K - 1);              // repeats the last direction past K
          const float* u = dirs + (size_t)k * 6;
#pragma unroll
          for (int c3 = 0; c3 < 3; ++c3) {
            uf[d][c3] = __ldg(u + c3);
            ut[d][c3] = __ldg(u + 3 + c3) * tscale;
          }
          h[d] = -INFINITY;
        }
        if (k_edges == 8)
          fold_contacts<true>(rec, np, way, ways, S.ce, S.se, sym, last, mu, uf, ut, h);
        else
          fold_contacts<false>(rec, np, way, ways, S.ce, S.se, sym, last, mu, uf, ut, h);
#pragma unroll
        for (int d = 0; d < kQD; ++d)
          if (k0 + d * groups < K) atomicMax(hmax + k0 + d * groups, float_order(h[d]));
      }
      if (tid == 0) S.total += nc;
      __syncthreads();
    }
    __syncthreads();
    float m = INFINITY;
    for (int k = tid; k < K; k += NT) m = fminf(m, order_float(hmax[k]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fminf(m, __shfl_xor_sync(kFull, m, o));
    if (lane == 0) S.red[warp] = m;
    __syncthreads();
    if (tid == 0) {
      float t = INFINITY;
#pragma unroll
      for (int w = 0; w < kQW; ++w) t = fminf(t, S.red[w]);
      eps[c] = t;
      if (ncontact) ncontact[c] = S.total;
    }
  }
  work_done(a.work);
}

template <class Kern>
cudaError_t grid_for_kernel(Kern k, size_t dyn, int B, int* grid) {
  int bps = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, k, kQW * 32, dyn);
  if (e != cudaSuccess) return e;
  if (bps < 1) bps = 1;
  long long g = (long long)device_sm_count() * bps;
  if (g > B) g = B;
  *grid = (int)g;
  return cudaSuccess;
}

}  // namespace

cudaError_t launch_contact_measure(const FusedArgs& a0, const float* weights, float tau, float* out, cudaStream_t st) {
  if (a0.B <= 0) return cudaSuccess;
  FusedArgs a = a0;
  cudaError_t ew = work_pair(&a.work, st);
  if (ew != cudaSuccess) return ew;
  int grid = 0;
  if (a.any_mesh) {
    cudaError_t e = grid_for_kernel(measure_kernel<true>, 0, a.B, &grid);
    if (e != cudaSuccess) return e;
    measure_kernel<true><<<grid, kQW * 32, 0, st>>>(a, weights, tau, out);
  } else {
    cudaError_t e = grid_for_kernel(measure_kernel<false>, 0, a.B, &grid);
    if (e != cudaSuccess) return e;
    measure_kernel<false><<<grid, kQW * 32, 0, st>>>(a, weights, tau, out);
  }
  return cudaGetLastError();
}

size_t epsilon_smem_bytes(int K) { return sizeof(ContactPair) * (kQBatch / 2) + sizeof(float) * (size_t)K; }

cudaError_t launch_grasp_epsilon(const FusedArgs& a0, float tau, float mu, int k_edges, float tscale,
                                 const float* dirs, int K, float* eps, int* ncontact, cudaStream_t st) {
  if (a0.B <= 0) return cudaSuccess;
  FusedArgs a = a0;
  cudaError_t ew = work_pair(&a.work, st);
  if (ew != cudaSuccess) return ew;
  const size_t dyn = epsilon_smem_bytes(K);
  static size_t attr_set[2][64] = {{0}, {0}};
  int dev = 0;
  cudaGetDevice(&dev);
  const int v = a.any_mesh ? 1 : 0;
  cudaError_t e = cudaSuccess;
  if (dyn > attr_set[v][dev & 63]) {
    e = a.any_mesh ? cudaFuncSetAttribute(epsilon_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn)
                   : cudaFuncSetAttribute(epsilon_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
    if (e != cudaSuccess) return e;
    attr_set[v][dev & 63] = dyn;
  }
  int grid = 0;
  if (a.any_mesh) {
    e = grid_for_kernel(epsilon_kernel<true>, dyn, a.B, &grid);
    if (e != cudaSuccess) return e;
    epsilon_kernel<true><<<grid, kQW * 32, dyn, st>>>(a, tau, mu, k_edges, tscale, dirs, K, eps, ncontact);
  } else {
    e = grid_for_kernel(epsilon_kernel<false>, dyn, a.B, &grid);
    if (e != cudaSuccess) return e;
    epsilon_kernel<false><<<grid, kQW * 32, dyn, st>>>(a, tau, mu, k_edges, tscale, dirs, K, eps, ncontact);
  }
  return cudaGetLastError();
}

}  // namespace fg
