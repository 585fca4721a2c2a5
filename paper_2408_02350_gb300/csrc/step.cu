// Per-step kernels of the meshfree BGK scheme (Sec. 3.2, 3.4.2, 5).
//
// k_transport_wp, k_transport_mirror, k_transport_batch (FP32 arithmetic; FP64 storage:
//   transport_f64.cu): one warp per interior point i.  The neighbour list and stencil of
//   i are staged in shared memory; for every neighbour j each lane reads f_j for its
//   velocities (16-byte loads) and accumulates
//     m_ij(v) = sum_d min(c.P_d, 0),  acc += m_ij f_j,  sk += m_ij,
//   with c = v - U_i^n (ALE) or v.  Since the upwind coefficient is
//   K_ij = sum_d (c.P_d - |c.P_d|) = 2 m_ij, the transported value is
//     f~_i = f_i - dt sum_j K_ij (f_j - f_i) = f_i - 2 dt (acc - sk f_i).
//   The same warp then sums the moments of f~_i over all velocities, forms rho, U, T,
//   tau and the Maxwellian, and writes f^{n+1} = (tau f~ + dt M)/(tau + dt) to the other
//   buffer: one read of f_i, neighbour reads served mostly from L1 and L2, one write.
// k_walls: one CTA per wall point; arriving velocities (v.n <= 0) get the WLS
//   reconstruction from interior f^{n+1}; leaving velocities get
//   rho_w M_w(v) with rho_w from zero net mass flux.
// k_move: x += dt U^{n+1} at interior points (FP64, no fused multiply-add).
#include <algorithm>
#include <type_traits>

#include "bgk_internal.cuh"
#include "device_common.cuh"
#include "motion.cuh"
#include "transport_wp.cuh"
#include "transport_stage.cuh"

namespace bgk {

static inline int grid_for(int64_t n, int block) { return (int)((n + block - 1) / block); }

__host__ __device__ static inline size_t align16(size_t b) { return (b + 15) & ~size_t(15); }

constexpr int RED_BYTES = 32 * 8 * 8;   // block-reduction scratch: 8 values x 32 warps, double
constexpr int NODE_BYTES = 64 * 8;      // velocity nodes, up to 64 per axis

// Finalise the moments from raw sums R = sum g, Mx = sum v g, E = sum |v|^2 g (+ sum h)
// (quadrature weight dv^dim applied to rho only; it cancels in U and T).
template <int DIM>
__device__ __forceinline__ void finish_moments(const double* tot, double wv, double* rho, double* U, double* T) {
  const double R = tot[0];
  double u2 = 0.0;
#pragma unroll
  for (int a = 0; a < DIM; ++a) { U[a] = tot[1 + a] / R; u2 += U[a] * U[a]; }
  *T = (tot[DIM + 1] - R * u2) / (3.0 * R);
  *rho = R * wv;
}

// Sum NVAL per-thread values: warp shuffles in T, then thread 0 adds the warp
// totals in double.  Result in out[] of every thread.
template <int NVAL, typename T>
__device__ __forceinline__ void block_sum0(const T (&v)[NVAL], double (&out)[NVAL], double* scratch) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarps = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int q = 0; q < NVAL; ++q) {
    T s = warp_sum(v[q]);
    if (lane == 0) scratch[q * 32 + warp] = (double)s;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int q = 0; q < NVAL; ++q) {
      double s = 0.0;
      for (int w = 0; w < nwarps; ++w) s += scratch[q * 32 + w];
      scratch[q * 32] = s;
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < NVAL; ++q) out[q] = scratch[q * 32];
  __syncthreads();
}

// Shared memory of the warp-per-point kernels with W warps: per warp the velocity nodes,
// the list and stencil, and (ks) the compensated moment sums.
template <int DIM>
__host__ __device__ inline size_t wp_smem_bytes(int W, int cap, bool ks = true) {
  return 256 * W + align16(sizeof(float) * list_floats<DIM>(cap) * W) + (ks ? sizeof(float) * kahan_floats<DIM>() * W : 0);
}
template <int DIM>
struct WarpShared {
  float* v;
  int32_t* col;
  float* P;
  float* k;
  __device__ __forceinline__ WarpShared(unsigned char* smem, int W, int warp, int cap) {
    v = reinterpret_cast<float*>(smem) + warp * 64;
    float* l = reinterpret_cast<float*>(smem + 256 * W);
    k = reinterpret_cast<float*>(smem + 256 * W + align16(sizeof(float) * list_floats<DIM>(cap) * W)) +
        warp * kahan_floats<DIM>();
    if (DIM == 2) {
      // 16-byte entries of all warps first, then the indices
      P = l + (size_t)warp * cap * 4;
      col = reinterpret_cast<int32_t*>(l + (size_t)W * cap * 4) + warp * cap;
    } else {
      P = l + (size_t)warp * list_floats<DIM>(cap);
      col = nullptr;
    }
  }
};

// Warps per CTA of the single-case first-order launch.  The CTA's points are consecutive
// in Morton order, but a smaller CTA loses less to the uneven neighbour counts of its
// warps (201^2 x 32^2 ALE cavity, transport ms: 1 warp 0.441, 2 0.440, 4 0.436, 8 0.440,
// 16 0.453, 32 0.503).
#ifndef BGK_WP_WARPS
#define BGK_WP_WARPS 4
#endif
// Warps per SM: 32 (64 registers); 28 (72 registers) for 2D BF16 with aligned velocity
// rows, whose conversions need them (201^2 x 32^2 ALE: 414 against 432 us per launch; FP32
// 411 against 406; ragged BF16, 190^2 x 30^2 ALE, two steps: 1069 against 1051 us); 16 with
// 8 velocities per lane.
template <typename S, int DIM, int VPL, bool ROW>
constexpr int wp_warps_per_sm() { return VPL != 4 ? 16 : (DIM == 2 && ROW && sizeof(S) == 2 ? 28 : 32); }
template <typename S, int DIM, bool ALE, bool ROW, int VPL, bool SH = false, bool AVG = false>
__global__ void __launch_bounds__(32 * BGK_WP_WARPS, wp_warps_per_sm<S, DIM, VPL, ROW>() / BGK_WP_WARPS)
    k_transport_wp(const CaseView cv) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int W = blockDim.x >> 5, warp = threadIdx.x >> 5;
  const WarpShared<DIM> ws(smem, W, warp, cv.cap);
  const int t = blockIdx.x * W + warp;
  if (t >= cv.n_int) return;
  transport_point_wp<S, DIM, ALE, ROW, VPL, VPL == 4, SH, AVG>(cv, cv.int_idx[t], ws.v, ws.col, ws.P, ws.k);
}

// Staged variant (2D, FP32, nv % 4 == 0): the neighbour rows come through per-warp rings
// of bulk copies instead of L1 (transport_stage.cuh).
#ifndef BGK_WP_STAGE
#define BGK_WP_STAGE 0
#endif
#ifndef BGK_STAGE_MINB
#define BGK_STAGE_MINB (32 / BGK_WP_WARPS)
#endif
template <bool ALE>
__global__ void __launch_bounds__(32 * BGK_WP_WARPS, BGK_STAGE_MINB) k_transport_stage(const CaseView cv) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int W = blockDim.x >> 5, warp = threadIdx.x >> 5;
  const int cap = cv.cap;
  const WarpShared<2> ws(smem, W, warp, cap);
  unsigned char* ring0 = smem + stage_ring_offset(wp_smem_bytes<2>(W, cap));
  float* s_ring = reinterpret_cast<float*>(ring0 + (size_t)warp * kStageD * kStageG * kStageRowBytes);
  uint64_t* s_bar = reinterpret_cast<uint64_t*>(ring0 + (size_t)W * kStageD * kStageG * kStageRowBytes) + warp * kStageD;
  const int t = blockIdx.x * W + warp;
  if (t >= cv.n_int) return;
  transport_point_stage<ALE>(cv, cv.int_idx[t], ws.v, ws.col, ws.P, ws.k, s_ring, s_bar);
}

// Second-order step, FP32/BF16 storage: one warp per interior point relaxes its output
// row exactly over dt/2 in place, with the moments of that row (compensated lane sums).
template <typename S, int DIM, bool ROW>
__global__ void __launch_bounds__(256) k_relax_half_wp(const CaseView cv) {
  constexpr int NC = DIM == 2 ? 2 : 1, VPL = 4;
  __shared__ __align__(16) float s_vall[8 * 64];  // chunk_velocities reads groups of 4
  const int W = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* s_v = s_vall + warp * 64;
  const int t = blockIdx.x * W + warp;
  if (t >= cv.n_int) return;
  for (int q = lane; q < cv.nv; q += 32) s_v[q] = cv.vnodes_f[q];
  __syncwarp();
  const int i = cv.int_idx[t];
  const int nv = cv.nv, NV = cv.NV, NVp = cv.NVp;
  const float inv_nv = 1.0f / (float)nv;
  const S* fi = reinterpret_cast<const S*>(cv.f_out) + (int64_t)i * NC * NVp;
  float msum[DIM + 2], mcmp[DIM + 2];
#pragma unroll
  for (int q = 0; q < DIM + 2; ++q) { msum[q] = 0.0f; mcmp[q] = 0.0f; }
  for (int chunk = lane; chunk * VPL < NVp; chunk += 32) {
    const int k0 = chunk * VPL;
    float vel[VPL][DIM];
    bool kin[VPL];
    chunk_velocities<DIM, VPL, ROW>(k0, nv, NV, inv_nv, s_v, vel, kin);
    float g[NC][VPL];
#pragma unroll
    for (int c = 0; c < NC; ++c) ldv<S, VPL>(fi + (int64_t)c * NVp + k0, g[c]);
    float ps[DIM + 2];
#pragma unroll
    for (int q = 0; q < DIM + 2; ++q) ps[q] = 0.0f;
#pragma unroll
    for (int e = 0; e < VPL; ++e) {
      const float g0 = kin[e] ? g[0][e] : 0.0f;
      float v2 = 0.0f;
      ps[0] += g0;
#pragma unroll
      for (int a = 0; a < DIM; ++a) { ps[1 + a] = fmaf(vel[e][a], g0, ps[1 + a]); v2 = fmaf(vel[e][a], vel[e][a], v2); }
      ps[DIM + 1] = fmaf(v2, g0, ps[DIM + 1]);
      if (NC == 2) ps[DIM + 1] += kin[e] ? g[NC - 1][e] : 0.0f;
    }
#pragma unroll
    for (int q = 0; q < DIM + 2; ++q) {
      const float y = ps[q] - mcmp[q];
      const float tt = msum[q] + y;
      mcmp[q] = (tt - msum[q]) - y;
      msum[q] = tt;
    }
  }
  finish_point<S, DIM, ROW, VPL, 1>(cv, i, s_v, msum, mcmp);
}

// Sharded step, FP32/BF16 storage: one warp per interior point relaxes f~ in the
// output row with the moments of the summed sums (the relaxation of k_transport_wp).
template <typename S, int DIM, bool ROW>
__global__ void __launch_bounds__(256) k_shard_relax_wp(const CaseView cv) {
  __shared__ __align__(16) float s_vall[8 * 64];  // chunk_velocities reads groups of 4
  const int W = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* s_v = s_vall + warp * 64;
  const int t = blockIdx.x * W + warp;
  if (t >= cv.n_int) return;
  for (int q = lane; q < cv.nv; q += 32) s_v[q] = cv.vnodes_f[q];
  __syncwarp();
  const int i = cv.int_idx[t];
  double tot[DIM + 2];
#pragma unroll
  for (int q = 0; q < DIM + 2; ++q) tot[q] = cv.xs[(int64_t)i * (DIM + 2) + q];
  relax_point<S, DIM, ROW, 4, true>(cv, i, s_v, tot);
}

// Fixed points with a mirror-symmetric velocity grid (nv % 4 == 0, NV % 8 == 0): one
// warp per interior point, each lane a velocity chunk and its mirror chunk; 128 registers,
// 16 warps per SM, five neighbours' rows in flight per warp (24 warps with 80 registers and
// two or three neighbours: 5.36 / 5.33 against 4.96 ms, 41^3 x 16^3).  Used in 3D, where it
// saves a quarter of the per-neighbour instructions; in 2D the extra registers cost about
// what the instructions save, and more in smaller clouds, so 2D keeps the plain kernel: step
// of 201^2 x 32^2 fixed points FP32 0.410 ms, paired 0.412 / 0.421 with 16 warps per SM and 5
// / 3 neighbours, 0.409 / 0.404 with 24 and 3 / 2, 0.438 with 32 and 2; 101^2 x 24^2 0.088
// against 0.094 ms at best (BF16 201^2 x 32^2: 0.423, paired 0.396 with 16 warps).
template <typename S, int DIM>
__global__ void __launch_bounds__(256, 2) k_transport_mirror(const CaseView cv) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int W = blockDim.x >> 5, warp = threadIdx.x >> 5;
  const WarpShared<DIM> ws(smem, W, warp, cv.cap);
  const int t = blockIdx.x * W + warp;
  if (t >= cv.n_int) return;
  transport_point_mirror<S, DIM>(cv, cv.int_idx[t], ws.v, ws.col, ws.P);
}

// Many cases in one persistent launch: items[k] = (case, interior slot), tiles of W
// consecutive items per CTA, tiles taken in grid-stride order.  Every warp reads
// its case's descriptor; the ROW4 variant is chosen per warp.
// 80 registers, 24 warps per SM (launched with 4 warps per CTA): a step of 24 cavities of up
// to 121^2 points takes 1409 us, 1743 with 16 warps, 1464 to 1580 with the compensated sums
// in shared memory (KS, as the single-case kernel), 1432 with 8 warps per CTA.
#ifndef BGK_BATCH_KS
#define BGK_BATCH_KS false
#endif
#ifndef BGK_BATCH_MIN_BLOCKS
#define BGK_BATCH_MIN_BLOCKS 3
#endif
template <typename S>
__global__ void __launch_bounds__(256, BGK_BATCH_MIN_BLOCKS) k_transport_batch(const CaseView* __restrict__ cases, const int2* __restrict__ items,
                                                             int n_items, int capmax) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int W = blockDim.x >> 5, warp = threadIdx.x >> 5;
  const WarpShared<2> ws(smem, W, warp, capmax);
  for (int tile = blockIdx.x; tile * W < n_items; tile += gridDim.x) {
    const int it = tile * W + warp;
    if (it >= n_items) continue;
    const int2 e = items[it];
    const CaseView& cv = cases[e.x];
    const int i = cv.int_idx[e.y];
    // (batched stepping takes fixed points only: c = v)
    if (cv.nv % 4 == 0) transport_point_wp<S, 2, false, true, 4, BGK_BATCH_KS>(cv, i, ws.v, ws.col, ws.P, ws.k);
    else transport_point_wp<S, 2, false, false, 4, BGK_BATCH_KS>(cv, i, ws.v, ws.col, ws.P, ws.k);
    __syncwarp();
  }
}

// Velocities per lane of moving points: 8 in 3D when the velocity rows split into groups of
// 8, whose rows cost fewer instructions per velocity and keep more loads in flight (first
// measured on fixed points, 41^3 x 16^3, which take the pairs now: 7.1 against 8.6 ms per
// step); 4 in 2D, where the lower occupancy of the wider variant costs more than it saves
// (201^2 x 32^2, at the time: 0.53 against 0.48 ms).
template <typename S, int DIM>
static void launch_transport_wp(const CaseView& cv, cudaStream_t s) {
  const int W = BGK_WP_WARPS, threads = 32 * W;
  const size_t smem = wp_smem_bytes<DIM>(W, cv.cap);
  const int grid = (cv.n_int + W - 1) / W;
  const bool row4 = cv.nv % 4 == 0;
  if constexpr (DIM == 3) {
    if (!cv.ale && row4) {  // (then NV % 8 == 0: the chunks of 4 pair up)
      auto k = k_transport_mirror<S, DIM>;
      const size_t msm = wp_smem_bytes<DIM>(W, cv.cap, false);
      cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)msm);
      k<<<grid, threads, msm, s>>>(cv);
      return;
    }
  }
  if constexpr (BGK_WP_STAGE && DIM == 2 && std::is_same<S, float>::value) {
    // (bulk copies need 16-byte aligned rows: caller-bound storage may start anywhere)
    if (row4 && cv.NVp % 4 == 0 && (reinterpret_cast<uintptr_t>(cv.f_in) & 15) == 0) {
      const size_t ssm = stage_smem_bytes(smem, W);
      auto k = cv.ale ? k_transport_stage<true> : k_transport_stage<false>;
      cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ssm);
      k<<<grid, threads, ssm, s>>>(cv);
      return;
    }
  }
#define BGK_LAUNCH_WP(ALE, ROW, VPL)                                                      \
  {                                                                                       \
    auto k = k_transport_wp<S, DIM, ALE, ROW, VPL>;                                       \
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);       \
    k<<<grid, threads, smem, s>>>(cv);                                                    \
  }
  if constexpr (DIM == 3) {
    if (!cv.ale) BGK_LAUNCH_WP(false, false, 4)
    else if (cv.nv % 8 == 0) BGK_LAUNCH_WP(true, true, 8)
    else if (row4) BGK_LAUNCH_WP(true, true, 4)
    else BGK_LAUNCH_WP(true, false, 4)
  } else if (cv.ale) {
    if (row4) BGK_LAUNCH_WP(true, true, 4) else BGK_LAUNCH_WP(true, false, 4)
  } else {
    if (row4) BGK_LAUNCH_WP(false, true, 4) else BGK_LAUNCH_WP(false, false, 4)
  }
#undef BGK_LAUNCH_WP
}

int launch_transport_fp32(const CaseView& cv, cudaStream_t s) {
  if (cv.n_int == 0) return 0;
  if (cv.dim == 2) {
    if (cv.storage == 1) launch_transport_wp<float, 2>(cv, s);
    else launch_transport_wp<__nv_bfloat16, 2>(cv, s);
  } else {
    if (cv.storage == 1) launch_transport_wp<float, 3>(cv, s);
    else launch_transport_wp<__nv_bfloat16, 3>(cv, s);
  }
  return 1;
}

template <typename S, int DIM>
static void launch_transport_avg_wp(const CaseView& cv, cudaStream_t s) {
  const int W = BGK_WP_WARPS, threads = 32 * W;
  const size_t smem = wp_smem_bytes<DIM>(W, cv.cap);
  const int grid = (cv.n_int + W - 1) / W;
  if (cv.nv % 4 == 0) {
    auto k = k_transport_wp<S, DIM, false, true, 4, false, true>;
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k<<<grid, threads, smem, s>>>(cv);
  } else {
    auto k = k_transport_wp<S, DIM, false, false, 4, false, true>;
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k<<<grid, threads, smem, s>>>(cv);
  }
}

int launch_transport_avg(const CaseView& cv, cudaStream_t s) {
  if (cv.n_int == 0) return 0;
  if (cv.storage == 0) return launch_transport_f64_avg(cv, s);
  if (cv.dim == 2) {
    if (cv.storage == 1) launch_transport_avg_wp<float, 2>(cv, s);
    else launch_transport_avg_wp<__nv_bfloat16, 2>(cv, s);
  } else {
    if (cv.storage == 1) launch_transport_avg_wp<float, 3>(cv, s);
    else launch_transport_avg_wp<__nv_bfloat16, 3>(cv, s);
  }
  return 1;
}

template <typename S, int DIM>
static void launch_relax_half_wp(const CaseView& cv, cudaStream_t s) {
  const int W = 8, grid = (cv.n_int + W - 1) / W;
  if (cv.nv % 4 == 0) k_relax_half_wp<S, DIM, true><<<grid, 32 * W, 0, s>>>(cv);
  else k_relax_half_wp<S, DIM, false><<<grid, 32 * W, 0, s>>>(cv);
}

int launch_relax_half(const CaseView& cv, cudaStream_t s) {
  if (cv.n_int == 0 || cv.tau_mode == 2) return 0;
  if (cv.storage == 0) return launch_relax_half_f64(cv, s);
  if (cv.dim == 2) {
    if (cv.storage == 1) launch_relax_half_wp<float, 2>(cv, s);
    else launch_relax_half_wp<__nv_bfloat16, 2>(cv, s);
  } else {
    if (cv.storage == 1) launch_relax_half_wp<float, 3>(cv, s);
    else launch_relax_half_wp<__nv_bfloat16, 3>(cv, s);
  }
  return 1;
}

int launch_transport(const CaseView& cv, cudaStream_t s) {
  if (cv.n_int == 0) return 0;
  if (cv.storage == 0) return launch_transport_f64(cv, s);
  if (cv.dim == 2) {
    if (cv.storage == 1) launch_transport_wp<float, 2>(cv, s);
    else launch_transport_wp<__nv_bfloat16, 2>(cv, s);
  } else {
    if (cv.storage == 1) launch_transport_wp<float, 3>(cv, s);
    else launch_transport_wp<__nv_bfloat16, 3>(cv, s);
  }
  return 1;
}

// ---------------------------------------------------------------------------
// walls
// ---------------------------------------------------------------------------
// The wall step of the sharded step (one CTA per wall point), split around the sum over all
// slabs (the whole step: walls_point_v4):
// PH = 1 writes the arriving half and the wall sums of the slab to cv.xs[w][2 dim + 6]
//   [0] sum_{arriving} |c_n| g   [1] sum_{leaving} c_n M_w   [2, dim + 4) moment sums of
//   the arriving half   [dim + 4, 2 dim + 6) moment sums of M_w over the leaving half;
// PH = 2 reads the summed cv.xs, writes rho_w M_w to the leaving half and the moments.
template <int DIM>
__host__ __device__ constexpr int wall_sums() { return 2 * DIM + 6; }

template <typename S, typename C, int DIM, int PH>
__device__ __forceinline__ void walls_point(const CaseView& cv, const int w, unsigned char* smem) {
  constexpr int NC = DIM == 2 ? 2 : 1;
  double* s_red = reinterpret_cast<double*>(smem);
  C* s_v = reinterpret_cast<C*>(smem + RED_BYTES);
  int32_t* s_j = reinterpret_cast<int32_t*>(smem + RED_BYTES + NODE_BYTES);
  C* s_r = reinterpret_cast<C*>(smem + RED_BYTES + NODE_BYTES + align16(sizeof(int32_t) * (cv.cap + 1)));
  const int b = cv.wall_idx[w];
  const int nv = cv.nv, NV = cv.NV, NVp = cv.NVp;
  const int vk0 = cv.vk0;
  if (PH == 1 && threadIdx.x < 32) {
    // warp 0 stages the interior neighbours in list order (ballot compaction)
    const int lane = threadIdx.x, m = checked_count(cv.cnt[b], cv.cap, cv.status);
    const int32_t* col = cv.col + (int64_t)b * cv.cap;
    const C* R = reinterpret_cast<const C*>(cv.recon) + (int64_t)b * cv.cap;
    int mi = 0;
    for (int s0 = 0; s0 < m; s0 += 32) {
      const int s = s0 + lane;
      const int j = s < m ? checked_index(col[s], cv.n, b, cv.status) : 0;
      const bool in = s < m && cv.kind[j] == 0;
      const unsigned bal = __ballot_sync(0xffffffffu, in);
      if (in) {
        const int pos = mi + __popc(bal & ((1u << lane) - 1u));
        s_j[1 + pos] = j;
        s_r[pos] = R[s];
      }
      mi += __popc(bal);
    }
    if (lane == 0) s_j[0] = mi;
  }
  for (int t = threadIdx.x; t < nv; t += blockDim.x) s_v[t] = (C)cv.vnodes[t];
  __syncthreads();
  const int mi = PH == 1 ? s_j[0] : 0;
  const int64_t rowlen = (int64_t)NC * NVp;
  S* f = reinterpret_cast<S*>(cv.f_out);
  S* fb = f + (int64_t)b * rowlen;
  const int8_t* cls = cv.wcls + (int64_t)w * NVp;
  const C* vn = reinterpret_cast<const C*>(cv.wvn) + (int64_t)w * NVp;
  const int kb = cv.kind[b];
  const int mrow = kb == cv.lid_wall ? 1 : (cv.body_wall > 0 && kb == cv.body_wall ? 2 : 0);
  const C* Mw = reinterpret_cast<const C*>(cv.mw) + (int64_t)mrow * NVp;
  const C cT = (C)cv.wall_T;

  // (PH 1) flux[0]: sum |c_n| g over the arriving half; flux[1]: sum c_n M_w over the
  // leaving half; part: moment sums of the arriving half; unit: those of M_w over the
  // leaving half
  C flux[2] = {(C)0, (C)0};
  C part[DIM + 2], unit[DIM + 2];
#pragma unroll
  for (int t = 0; t < DIM + 2; ++t) { part[t] = (C)0; unit[t] = (C)0; }
  if (PH == 1) {
    for (int k = threadIdx.x; k < NV; k += blockDim.x) {
      if (cls[k] == 0) {
        C g[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) g[c] = (C)0;
        for (int s = 0; s < mi; ++s) {
          const S* fj = f + (int64_t)s_j[1 + s] * rowlen;
          const C r = s_r[s];
#pragma unroll
          for (int c = 0; c < NC; ++c) g[c] += r * ld1(fj + (int64_t)c * NVp + k);
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) st1(fb + (int64_t)c * NVp + k, g[c]);
        flux[0] += vn[k] * g[0];
        int kk = k + vk0;
        C v2 = (C)0;
        part[0] += g[0];
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
          const C va = s_v[kk % nv];
          kk /= nv;
          part[1 + a] += va * g[0];
          v2 += va * va;
        }
        part[DIM + 1] += v2 * g[0];
        if (NC == 2) part[DIM + 1] += g[NC - 1];
      } else {
        const C m0 = Mw[k];
        flux[1] += vn[k] * m0;
        int kk = k + vk0;
        C v2 = (C)0;
        unit[0] += m0;
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
          const C va = s_v[kk % nv];
          kk /= nv;
          unit[1 + a] += va * m0;
          v2 += va * va;
        }
        unit[DIM + 1] += v2 * m0;
        if (NC == 2) unit[DIM + 1] += cT * m0;
      }
    }
  }
  if constexpr (PH == 1) {
    double t1[DIM + 4], t2[DIM + 2];
    C v1[DIM + 4];
    v1[0] = flux[0];
    v1[1] = flux[1];
#pragma unroll
    for (int q = 0; q < DIM + 2; ++q) v1[2 + q] = part[q];
    block_sum0<DIM + 4, C>(v1, t1, s_red);
    block_sum0<DIM + 2, C>(unit, t2, s_red);
    if (threadIdx.x == 0) {
      double* xw = cv.xs + (int64_t)w * wall_sums<DIM>();
#pragma unroll
      for (int q = 0; q < DIM + 4; ++q) xw[q] = t1[q];
#pragma unroll
      for (int q = 0; q < DIM + 2; ++q) xw[DIM + 4 + q] = t2[q];
    }
    return;
  }
  const double* xw = cv.xs + (int64_t)w * wall_sums<DIM>();
  const double rho_w = xw[0] / xw[1];
  const C crw = (C)rho_w;
  for (int k = threadIdx.x; k < NV; k += blockDim.x) {
    if (cls[k] != 0) {
      const C g0 = crw * Mw[k];
      st1(fb + k, g0);
      if (NC == 2) st1(fb + NVp + k, cT * g0);
    }
  }
  double tot[DIM + 2];
#pragma unroll
  for (int q = 0; q < DIM + 2; ++q) tot[q] = xw[2 + q] + rho_w * xw[DIM + 4 + q];
  if (threadIdx.x == 0) {
    double rho, Un[3] = {0, 0, 0}, T;
    const double wv = cv.wv;
    finish_moments<DIM>(tot, wv, &rho, Un, &T);
    double* mo = cv.mom + (int64_t)b * MOM_STRIDE;
    mo[0] = rho; mo[1] = Un[0]; mo[2] = Un[1]; mo[3] = Un[2]; mo[4] = T;
    if (!(rho_w >= 0.0) || !isfinite(rho_w)) set_status(cv.status, ST_NONFINITE);
  }
}

// The whole wall step of one wall point by one CTA, 4 consecutive velocities per thread and
// access.  Bound by latency (a wall point reads about 8 rows, and a cavity has one wall
// point per lattice point of its boundary), so the chain of dependent steps is short:
//   - warp 0 compacts the neighbours with a non-zero weight (wall neighbours have weight
//     zero), so the kinds of the neighbours are not read;
//   - one reduction: the arriving flux and the arriving half's moment sums together; the
//     leaving half's moments are rho_w times the sums of M_w tabulated per wall point
//     (wunit), so they need no second reduction;
//   - velocity indices split by one float quotient per 4 velocities where a grid row holds
//     them (ROW), without integer divisions.
// 160 wall points x 256 velocities (41^2 cavity) 11.6 us with two reductions and a scalar
// velocity per thread (2D; FP64 15.5 us), 7464 wall points of 24 cavities 123 us.
// Threads from wall_threads(NVp) on only take part in the barriers, so a wider launch
// (the batched one) computes the same bits.
__host__ __device__ inline int wall_threads(int NVp) {
  const int t = (NVp / 4 + 31) / 32 * 32;
  return t < 256 ? t : 256;
}

template <typename C> struct WallNodes;
template <> struct WallNodes<float> {
  static __device__ __forceinline__ const float* of(const CaseView& cv) { return cv.vnodes_f; }
};
template <> struct WallNodes<double> {
  static __device__ __forceinline__ const double* of(const CaseView& cv) { return cv.vnodes; }
};

// Shared memory of the body: neighbours and weights [cap], nodes [64], sums [8 warps][8],
// rho_w, the neighbour count.
__host__ __device__ inline size_t wall_smem(int cap) {
  return align16(sizeof(double) * (size_t)cap) + align16(sizeof(int32_t) * cap) + 64 * 8 + 64 * 8 + 16;
}

template <typename S, typename C, int DIM>
__device__ __forceinline__ void walls_point_v4(const CaseView& cv, const int w, unsigned char* smem) {
  constexpr int NC = DIM == 2 ? 2 : 1, NS = DIM + 3;
  const int cap = cv.cap;
  C* s_r = reinterpret_cast<C*>(smem);
  unsigned char* q0 = smem + align16(sizeof(double) * (size_t)cap);
  int32_t* s_j = reinterpret_cast<int32_t*>(q0);
  q0 += align16(sizeof(int32_t) * cap);
  C* s_v = reinterpret_cast<C*>(q0);
  C* s_sum = reinterpret_cast<C*>(q0 + 512);
  double* s_rho = reinterpret_cast<double*>(q0 + 1024);
  int32_t* s_mi = reinterpret_cast<int32_t*>(q0 + 1032);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = cv.wall_idx[w];
  const int nv = cv.nv, NV = cv.NV, NVp = cv.NVp, nchunk = NVp >> 2;
  const int T = wall_threads(NVp);
  if (tid < 32) {
    const int m = checked_count(cv.cnt[b], cap, cv.status);
    const int32_t* col = cv.col + (int64_t)b * cap;
    const C* R = reinterpret_cast<const C*>(cv.recon) + (int64_t)b * cap;
    int mi = 0;
    for (int s0 = 0; s0 < m; s0 += 32) {
      const int s = s0 + lane;
      const int j = s < m ? checked_index(col[s], cv.n, b, cv.status) : 0;
      const C r = s < m ? R[s] : (C)0;
      const unsigned bal = __ballot_sync(0xffffffffu, r != (C)0);
      if (r != (C)0) {
        const int pos = mi + __popc(bal & ((1u << lane) - 1u));
        s_j[pos] = j;
        s_r[pos] = r;
      }
      mi += __popc(bal);
    }
    if (lane == 0) *s_mi = mi;
  }
  for (int t = tid; t < nv; t += blockDim.x) s_v[t] = WallNodes<C>::of(cv)[t];
  __syncthreads();
  const int mi = *s_mi;
  const int64_t rowlen = (int64_t)NC * NVp;
  S* f = reinterpret_cast<S*>(cv.f_out);
  S* fb = f + (int64_t)b * rowlen;
  const int8_t* cls = cv.wcls + (int64_t)w * NVp;
  const C* vn = reinterpret_cast<const C*>(cv.wvn) + (int64_t)w * NVp;
  const float inv_nv = 1.0f / (float)nv;
  const bool row = nv % 4 == 0;

  // sums over the arriving half: flux, sum g, sum v g, sum |v|^2 g (+ sum h)
  C sum[NS];
#pragma unroll
  for (int t = 0; t < NS; ++t) sum[t] = (C)0;
  for (int ch = tid; ch < nchunk; ch += T) {
    if (tid >= T) break;
    const int k0 = 4 * ch;
    const char4 c4 = *reinterpret_cast<const char4*>(cls + k0);
    const bool arr[4] = {c4.x == 0 && k0 < NV, c4.y == 0 && k0 + 1 < NV, c4.z == 0 && k0 + 2 < NV,
                         c4.w == 0 && k0 + 3 < NV};
    if (!(arr[0] || arr[1] || arr[2] || arr[3])) continue;
    C g[NC][4];
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
      for (int e = 0; e < 4; ++e) g[c][e] = (C)0;
#pragma unroll 4
    for (int s = 0; s < mi; ++s) {
      const S* fj = f + (int64_t)s_j[s] * rowlen + k0;
      const C r = s_r[s];
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        C v[4];
        ld4(fj + (int64_t)c * NVp, v);
#pragma unroll
        for (int e = 0; e < 4; ++e) g[c][e] += r * v[e];
      }
    }
    C vnv[4];
    ld4(vn + k0, vnv);
    int ia[4][DIM];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      if (row && e > 0) {
#pragma unroll
        for (int a = 0; a < DIM; ++a) ia[e][a] = ia[0][a] + (a == 0 ? e : 0);
      } else {
        int kk = k0 + e < NV ? k0 + e : 0;
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
          const int q = fdiv_small(kk, inv_nv);
          ia[e][a] = kk - q * nv;
          kk = q;
        }
      }
    }
    if (arr[0] && arr[1] && arr[2] && arr[3]) {
#pragma unroll
      for (int c = 0; c < NC; ++c) st4(fb + (int64_t)c * NVp + k0, g[c]);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      if (!arr[e]) continue;
      if (!(arr[0] && arr[1] && arr[2] && arr[3])) {
#pragma unroll
        for (int c = 0; c < NC; ++c) st1(fb + (int64_t)c * NVp + k0 + e, g[c][e]);
      }
      const C g0 = g[0][e];
      sum[0] += vnv[e] * g0;
      sum[1] += g0;
      C v2 = (C)0;
#pragma unroll
      for (int a = 0; a < DIM; ++a) {
        const C va = s_v[ia[e][a]];
        sum[2 + a] += va * g0;
        v2 += va * va;
      }
      sum[DIM + 2] += v2 * g0;
      if (NC == 2) sum[DIM + 2] += g[NC - 1][e];
    }
  }
#pragma unroll
  for (int t = 0; t < NS; ++t) {
    const C x = warp_sum(sum[t]);
    if (lane == 0) s_sum[warp * 8 + t] = x;
  }
  __syncthreads();
  if (tid < 32) {
    // lane t: the total of sum t over the warps, in FP64
    double tot = 0.0;
    if (lane < NS)
      for (int q = 0; q < (T >> 5); ++q) tot += (double)s_sum[q * 8 + lane];
    const double rho_w = __shfl_sync(0xffffffffu, tot, 0) * cv.winv[w];
    if (lane == 0) *s_rho = rho_w;
    const double all = lane >= 1 && lane < NS ? fma(rho_w, cv.wunit[(int64_t)w * (DIM + 2) + lane - 1], tot) : 0.0;
    double m[DIM + 2];
#pragma unroll
    for (int q = 0; q < DIM + 2; ++q) m[q] = __shfl_sync(0xffffffffu, all, q + 1);
    if (lane == 0) {
      double rho, Un[3] = {0, 0, 0}, Tn;
      finish_moments<DIM>(m, cv.wv, &rho, Un, &Tn);
      double* mo = cv.mom + (int64_t)b * MOM_STRIDE;
      mo[0] = rho; mo[1] = Un[0]; mo[2] = Un[1]; mo[3] = Un[2]; mo[4] = Tn;
      if (!(rho_w >= 0.0) || !isfinite(rho_w)) set_status(cv.status, ST_NONFINITE);
    }
  }
  __syncthreads();
  const int kb = cv.kind[b];
  const int mrow = kb == cv.lid_wall ? 1 : (cv.body_wall > 0 && kb == cv.body_wall ? 2 : 0);
  const C* Mw = reinterpret_cast<const C*>(cv.mw) + (int64_t)mrow * NVp;
  const C crw = (C)*s_rho, cT = (C)cv.wall_T;
  for (int ch = tid; ch < nchunk; ch += T) {
    if (tid >= T) break;
    const int k0 = 4 * ch;
    const char4 c4 = *reinterpret_cast<const char4*>(cls + k0);
    const bool lv[4] = {c4.x != 0, c4.y != 0, c4.z != 0, c4.w != 0};
    if (!(lv[0] || lv[1] || lv[2] || lv[3])) continue;
    C g[4], h[4];
    ld4(Mw + k0, g);
#pragma unroll
    for (int e = 0; e < 4; ++e) { g[e] = crw * g[e]; h[e] = cT * g[e]; }
    if (lv[0] && lv[1] && lv[2] && lv[3]) {
      st4(fb + k0, g);
      if (NC == 2) st4(fb + NVp + k0, h);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (lv[e]) {
          st1(fb + k0 + e, g[e]);
          if (NC == 2) st1(fb + NVp + k0 + e, h[e]);
        }
    }
  }
}

template <typename S, typename C, int DIM>
__global__ void __launch_bounds__(256) k_walls_v4(const CaseView cv) {
  extern __shared__ __align__(16) unsigned char smem[];
  walls_point_v4<S, C, DIM>(cv, blockIdx.x, smem);
}

template <typename S, typename C, int DIM, int PH>
__global__ void __launch_bounds__(256) k_walls(const CaseView cv) {
  extern __shared__ __align__(16) unsigned char smem[];
  walls_point<S, C, DIM, PH>(cv, blockIdx.x, smem);
}

// witems[k] = (case, wall slot): one CTA per wall point of any case
template <typename S, typename C>
__global__ void __launch_bounds__(256) k_walls_batch(const CaseView* __restrict__ cases, const int2* __restrict__ witems) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int2 e = witems[blockIdx.x];
  walls_point_v4<S, C, 2>(cases[e.x], e.y, smem);
}

int launch_transport_batch(const CaseView* d_cases, const int2* items, int n_items, int storage, int capmax,
                           int warps, int grid, cudaStream_t s) {
  if (n_items == 0) return 0;
  const int threads = 32 * warps;
  const size_t smem = wp_smem_bytes<2>(warps, capmax);
  const int ntiles = (n_items + warps - 1) / warps;
  if (grid <= 0 || grid > ntiles) grid = ntiles;
  auto go = [&](auto k) {
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k<<<grid, threads, smem, s>>>(d_cases, items, n_items, capmax);
  };
  if (storage == 1) go(k_transport_batch<float>);
  else go(k_transport_batch<__nv_bfloat16>);
  return 1;
}

int launch_walls_batch(const CaseView* d_cases, const int2* witems, int n_witems, int storage, int capmax,
                       int nvpmax, cudaStream_t s) {
  if (n_witems == 0) return 0;
  const size_t smem = wall_smem(capmax);
  const int threads = wall_threads(nvpmax);
  if (storage == 1) k_walls_batch<float, float><<<n_witems, threads, smem, s>>>(d_cases, witems);
  else k_walls_batch<__nv_bfloat16, float><<<n_witems, threads, smem, s>>>(d_cases, witems);
  return 1;
}

int launch_walls(const CaseView& cv, cudaStream_t s) {
  if (cv.n_wall == 0) return 0;
  const int threads = wall_threads(cv.NVp);
  const size_t smem = wall_smem(cv.cap);
  if (cv.dim == 2) {
    if (cv.storage == 0) k_walls_v4<double, double, 2><<<cv.n_wall, threads, smem, s>>>(cv);
    else if (cv.storage == 1) k_walls_v4<float, float, 2><<<cv.n_wall, threads, smem, s>>>(cv);
    else k_walls_v4<__nv_bfloat16, float, 2><<<cv.n_wall, threads, smem, s>>>(cv);
  } else {
    if (cv.storage == 0) k_walls_v4<double, double, 3><<<cv.n_wall, threads, smem, s>>>(cv);
    else if (cv.storage == 1) k_walls_v4<float, float, 3><<<cv.n_wall, threads, smem, s>>>(cv);
    else k_walls_v4<__nv_bfloat16, float, 3><<<cv.n_wall, threads, smem, s>>>(cv);
  }
  return 1;
}

// ---------------------------------------------------------------------------
// wall tables: classification by the normal velocity relative to the wall,
// c_n = (v - u_w).n, |c_n|, 1/sum_{c_n>0} c_n M_w and the unit-density wall
// Maxwellians, all evaluated in FP64.  u_w is lid_u on the lid, body_u on the
// body, zero elsewhere; the tables stay valid while the walls translate.
// ---------------------------------------------------------------------------
__device__ __forceinline__ const double* wall_velocity(const CaseView& cv, int kb, const double* zero) {
  if (kb == cv.lid_wall) return cv.lid_u;
  if (cv.body_wall > 0 && kb == cv.body_wall) return cv.body_u;
  return zero;
}

template <typename C, int DIM>
__global__ void __launch_bounds__(256) k_wall_tables(CaseView cv) {
  constexpr int NS = DIM + 3;
  __shared__ double s_sum[8][NS];
  const int w = blockIdx.x;
  const int b = cv.wall_idx[w];
  const int nv = cv.nv, NV = cv.NV, NVp = cv.NVp;
  double nb[DIM];
#pragma unroll
  for (int a = 0; a < DIM; ++a) nb[a] = cv.normal[(int64_t)b * DIM + a];
  const double zero[3] = {0.0, 0.0, 0.0};
  const double* uw = wall_velocity(cv, cv.kind[b], zero);
  const double pi = 3.14159265358979323846, T = cv.wall_T;
  const double pref = DIM == 2 ? 1.0 / (2.0 * pi * T) : 1.0 / pow(2.0 * pi * T, 1.5);
  // sum_{c_n > 0} c_n M_w, then the moment sums of the stored M_w over those velocities
  double acc[NS];
#pragma unroll
  for (int t = 0; t < NS; ++t) acc[t] = 0.0;
  for (int k = threadIdx.x; k < NVp; k += blockDim.x) {
    int8_t cl = 0;
    double avn = 0.0;
    if (k < NV) {
      int kk = k + cv.vk0;
      double vn = 0.0, c2 = 0.0, vv[DIM];
#pragma unroll
      for (int a = 0; a < DIM; ++a) {
        const double va = cv.vnodes[kk % nv];
        vv[a] = va;
        kk /= nv;
        const double c = __dadd_rn(va, -uw[a]);
        vn = __dadd_rn(vn, __dmul_rn(c, nb[a]));
        c2 += c * c;
      }
      cl = vn > 0.0 ? 1 : 0;
      avn = fabs(vn);
      if (cl) {
        const double M = pref * exp(-c2 / (2.0 * T)), m0 = (double)(C)M;
        acc[0] += vn * M;
        acc[1] += m0;
        double v2 = 0.0;
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
          acc[2 + a] += vv[a] * m0;
          v2 += vv[a] * vv[a];
        }
        acc[DIM + 2] += v2 * m0;
        if (DIM == 2) acc[DIM + 2] += T * m0;
      }
    }
    cv.wcls[(int64_t)w * NVp + k] = cl;
    reinterpret_cast<C*>(cv.wvn)[(int64_t)w * NVp + k] = (C)avn;
  }
#pragma unroll
  for (int t = 0; t < NS; ++t) {
    const double x = warp_sum(acc[t]);
    if ((threadIdx.x & 31) == 0) s_sum[threadIdx.x >> 5][t] = x;
  }
  __syncthreads();
  if (threadIdx.x >= 1 && threadIdx.x < NS) {
    double t = 0.0;
    for (int q = 0; q < (int)(blockDim.x + 31) / 32; ++q) t += s_sum[q][threadIdx.x];
    cv.wunit[(int64_t)w * (DIM + 2) + threadIdx.x - 1] = t;
  }
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int q = 0; q < (int)(blockDim.x + 31) / 32; ++q) s += s_sum[q][0];
    // a velocity slab of a sharded case holds part of this sum (its wall step takes
    // the sum over all slabs instead): no check there
    const bool slab = cv.vk0 != 0 || NV != (DIM == 2 ? nv * nv : nv * nv * nv);
    cv.winv[w] = s > 0.0 ? 1.0 / s : 0.0;
    if (!(s > 0.0) && !slab) set_status(cv.status, ST_SINGULAR);
  }
}

template <typename C, int DIM>
__global__ void k_mw_table(CaseView cv) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= cv.NVp) return;
  const double pi = 3.14159265358979323846, T = cv.wall_T;
  const double pref = DIM == 2 ? 1.0 / (2.0 * pi * T) : 1.0 / pow(2.0 * pi * T, 1.5);
  const double zero[3] = {0.0, 0.0, 0.0};
  for (int row = 0; row < 3; ++row) {
    const double* uw = row == 0 ? zero : (row == 1 ? cv.lid_u : cv.body_u);
    double M = 0.0;
    if (k < cv.NV) {
      int kk = k + cv.vk0;
      double c2 = 0.0;
      for (int a = 0; a < DIM; ++a) {
        const double c = cv.vnodes[kk % cv.nv] - uw[a];
        kk /= cv.nv;
        c2 += c * c;
      }
      M = pref * exp(-c2 / (2.0 * T));
    }
    reinterpret_cast<C*>(cv.mw)[row * cv.NVp + k] = (C)M;
  }
}

// Velocity nodes v_j = -vmax + j dv in the centred form (j - (nv-1)/2) dv, exactly
// symmetric about zero (Sec. 3.3).
__global__ void k_nodes(CaseView cv) {
  const int j = threadIdx.x;
  if (j < cv.nv) {
    const double v = __dmul_rn(__dadd_rn((double)j, -0.5 * (double)(cv.nv - 1)), cv.dv);
    cv.vnodes[j] = v;
    cv.vnodes_f[j] = (float)v;
  }
}

int launch_init_tables(const CaseView& cv, cudaStream_t s) {
  int n = 1;
  k_nodes<<<1, 64, 0, s>>>(cv);
  const bool f64 = cv.storage == 0;
  if (cv.dim == 2) {
    if (f64) k_mw_table<double, 2><<<grid_for(cv.NVp, 256), 256, 0, s>>>(cv);
    else k_mw_table<float, 2><<<grid_for(cv.NVp, 256), 256, 0, s>>>(cv);
  } else {
    if (f64) k_mw_table<double, 3><<<grid_for(cv.NVp, 256), 256, 0, s>>>(cv);
    else k_mw_table<float, 3><<<grid_for(cv.NVp, 256), 256, 0, s>>>(cv);
  }
  ++n;
  if (cv.n_wall > 0) {
    if (cv.dim == 2) {
      if (f64) k_wall_tables<double, 2><<<cv.n_wall, 256, 0, s>>>(cv);
      else k_wall_tables<float, 2><<<cv.n_wall, 256, 0, s>>>(cv);
    } else {
      if (f64) k_wall_tables<double, 3><<<cv.n_wall, 256, 0, s>>>(cv);
      else k_wall_tables<float, 3><<<cv.n_wall, 256, 0, s>>>(cv);
    }
    ++n;
  }
  return n;
}

// ---------------------------------------------------------------------------
// point motion (Eqs. originalALE1, ALE1)
// ---------------------------------------------------------------------------
// After every CTA has read the body centre and merged its maximum squared
// displacement (bits b) into disp2, the last one decides whether the next list
// build rebuilds the candidates and advances the centre to cn.
__device__ __forceinline__ void move_merge(const CaseView& cv, uint32_t b, double thr2, const double* cn) {
  if (cv.sk) atomicMax(&cv.sk->disp2, b);
  __threadfence();
  uint32_t* ctr = cv.sk ? &cv.sk->blocks : &cv.body->blocks;
  if (atomicAdd(ctr, 1u) == gridDim.x - 1) {
    __threadfence();
    if (cv.sk) {
      const uint32_t d = atomicOr(&cv.sk->disp2, 0u);
      const int rb = (double)__uint_as_float(d) > thr2;
      cv.sk->rebuild = rb;
      if (rb) cv.sk->disp2 = 0u;
    }
    if (cv.body)
      for (int a = 0; a < cv.dim; ++a) cv.body->c[a] = cn[a];
    *ctr = 0u;
  }
}

// Threads [0, n_int) move the interior points, threads [n_int, n_int + n_wall) the
// body's boundary points among the wall points (when there is a body).  With skin
// lists the kernel also tracks max |x - x_b|^2; its last CTA decides whether the next
// list build rebuilds the candidates (max |x - x_b| > h skin / 2, thr2 = (h skin /
// 2)^2 (1 - 1e-6)) and advances the body centre.
__global__ void __launch_bounds__(256) k_move(CaseView cv, double thr2) {
  __shared__ uint32_t s_max[8];
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  double cn[3];
  body_centre_next(cv, cn);
  const double d2 = move_thread(cv, t, cn);
  if (cv.sk || cv.body) {
    // CTA maximum of the displacement bits (non-negative floats order as integers)
    const uint32_t w = __reduce_max_sync(0xffffffffu, __float_as_uint(__double2float_ru(d2)));
    if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = w;
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t b = 0;
      for (int k = 0; k < (int)(blockDim.x >> 5); ++k) b = max(b, s_max[k]);
      move_merge(cv, b, thr2, cn);
    }
  }
}

int launch_move(const CaseView& cv, cudaStream_t s) {
  const int64_t n = (int64_t)cv.n_int + (cv.body ? cv.n_wall : 0);
  if (n == 0) return 0;
  const double half = 0.5 * cv.h * cv.skin;
  k_move<<<grid_for(n, 256), 256, 0, s>>>(cv, half * half * (1.0 - 1e-6));
  return 1;
}

// ---------------------------------------------------------------------------
// initial Maxwellian, moments of a given f, layout conversion
// ---------------------------------------------------------------------------
// The same Maxwellian at every point: thread k of column block y evaluates M(v_k) once and
// writes it (and T0 M, the Chu h component) into the rows of the points of its block
// (blockIdx.x, blockIdx.x + gridDim.x, ...), so that a grid of a few hundred blocks
// evaluates a few hundred rows' worth of exponentials, not one per (point, velocity).
template <typename S, int DIM>
__global__ void k_set_maxwellian(CaseView cv, double rho0, double u0, double u1, double u2, double T0) {
  constexpr int NC = DIM == 2 ? 2 : 1;
  const int k = blockIdx.y * blockDim.x + threadIdx.x;
  if (k >= cv.NVp) return;
  const double pi = 3.14159265358979323846;
  double M = 0.0;
  if (k < cv.NV) {
    const double U[3] = {u0, u1, u2};
    int kk = k + cv.vk0;
    double c2 = 0.0;
    for (int a = 0; a < DIM; ++a) {
      const double c = cv.vnodes[kk % cv.nv] - U[a];
      kk /= cv.nv;
      c2 += c * c;
    }
    const double pref = DIM == 2 ? rho0 / (2.0 * pi * T0) : rho0 / pow(2.0 * pi * T0, 1.5);
    M = pref * exp(-c2 / (2.0 * T0));
  }
  using C = decltype(ld1(reinterpret_cast<const S*>(cv.f_in)));
  const C m0 = (C)M, m1 = (C)(T0 * M);
  for (int i = blockIdx.x; i < cv.n; i += gridDim.x) {
    S* f = reinterpret_cast<S*>(cv.f_in) + (int64_t)i * NC * cv.NVp;
    st1(f + k, m0);
    if (NC == 2) st1(f + cv.NVp + k, m1);
  }
}

int launch_set_maxwellian(const CaseView& cv, double rho0, const double* u0, double T0, cudaStream_t s) {
  const dim3 g((unsigned)std::min(cv.n, 1216), (unsigned)((cv.NVp + 255) / 256));
  if (cv.dim == 2) {
    if (cv.storage == 0) k_set_maxwellian<double, 2><<<g, 256, 0, s>>>(cv, rho0, u0[0], u0[1], 0.0, T0);
    else if (cv.storage == 1) k_set_maxwellian<float, 2><<<g, 256, 0, s>>>(cv, rho0, u0[0], u0[1], 0.0, T0);
    else k_set_maxwellian<__nv_bfloat16, 2><<<g, 256, 0, s>>>(cv, rho0, u0[0], u0[1], 0.0, T0);
  } else {
    if (cv.storage == 0) k_set_maxwellian<double, 3><<<g, 256, 0, s>>>(cv, rho0, u0[0], u0[1], u0[2], T0);
    else if (cv.storage == 1) k_set_maxwellian<float, 3><<<g, 256, 0, s>>>(cv, rho0, u0[0], u0[1], u0[2], T0);
    else k_set_maxwellian<__nv_bfloat16, 3><<<g, 256, 0, s>>>(cv, rho0, u0[0], u0[1], u0[2], T0);
  }
  return 1;
}

// Moments of every point of f (internal layout), one CTA per point.  SH: the raw sums
// of the velocity slab to the exchange buffer instead.
template <typename S, typename C, int DIM, bool SH = false>
__global__ void k_moments(CaseView cv, const S* f) {
  constexpr int NC = DIM == 2 ? 2 : 1;
  __shared__ double s_red[8 * 32];
  const int i = blockIdx.x;
  const int nv = cv.nv, NV = cv.NV, NVp = cv.NVp;
  const S* fi = f + (int64_t)i * NC * NVp;
  C part[DIM + 2];
#pragma unroll
  for (int t = 0; t < DIM + 2; ++t) part[t] = (C)0;
  for (int k = threadIdx.x; k < NV; k += blockDim.x) {
    const C g = ld1(fi + k);
    int kk = k + (SH ? cv.vk0 : 0);
    C v2 = (C)0;
    part[0] += g;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      const C va = (C)cv.vnodes[kk % nv];
      kk /= nv;
      part[1 + a] += va * g;
      v2 += va * va;
    }
    part[DIM + 1] += v2 * g;
    if (NC == 2) part[DIM + 1] += ld1(fi + NVp + k);
  }
  double tot[DIM + 2];
  block_sum0<DIM + 2, C>(part, tot, s_red);
  if (SH && threadIdx.x == 0) {
#pragma unroll
    for (int q = 0; q < DIM + 2; ++q) cv.xs[(int64_t)i * (DIM + 2) + q] = tot[q];
  } else if (threadIdx.x == 0) {
    double rho, Un[3] = {0, 0, 0}, T;
    const double wv = cv.wv;
    finish_moments<DIM>(tot, wv, &rho, Un, &T);
    double* mo = cv.mom + (int64_t)i * MOM_STRIDE;
    mo[0] = rho; mo[1] = Un[0]; mo[2] = Un[1]; mo[3] = Un[2]; mo[4] = T;
  }
}

// FP32/BF16 storage: each warp streams gp consecutive points in turn, each lane 4
// consecutive velocities per chunk (16-byte loads, eight chunks in flight, velocity nodes
// staged in shared memory as FP32) into Kahan-compensated FP32 sums.  A point's lane sums
// are reduced across the warp as FP32 pairs with exact high-part additions (no FP64 on
// the 32-lane path); once the CTA has all its points, thread t converts point t's pair
// totals to FP64 and forms rho, U, T in FP64, so each FP64 instruction serves up to 32
// points (FP64 runs at a small fraction of the FP32 rate, whatever the lanes in use).  SH:
// the raw sums of the velocity slab (in FP64) to the exchange buffer instead.  48 registers
// (5 CTAs per SM), chosen so that the loads of a chunk stay in flight (left to the compiler,
// 40 for BF16: 35 against 29 us, 41^2 x 63^2).
constexpr int MOM_GP = 4, MOM_WARPS = 8;  // points per warp, warps per CTA (at most)
// Points per warp: MOM_GP (32 points per CTA, one full warp of FP64 work) where that still
// gives every SM 32 warps, fewer for smaller clouds; 8 left the last CTAs uneven (201^2 x
// 32^2, upload and moments: 161 us, 166 with 32-point CTAs of 4 warps).
static int moments_gp(int n) { return std::max(1, std::min(MOM_GP, n / (TARGET_SMS * 32))); }
// Warps per CTA: 8, so that the FP64 part serves 8 points or more at once (21^3 points x 3^3
// velocities, upload and moments: 17 us; 39 us with a warp for each point's FP64 part, 20 us
// with 4 warps of 8 points); 4 where the warps do not fill the SMs and 8 would spread them
// unevenly.
static int moments_warps(int n) { return n < TARGET_SMS * 32 ? MOM_WARPS / 2 : MOM_WARPS; }
template <typename S, int DIM, bool ROW, bool SH = false>
__global__ void __launch_bounds__(32 * MOM_WARPS, 5) k_moments_wp(CaseView cv, const S* f, const int gp) {
  constexpr int NC = DIM == 2 ? 2 : 1, VPL = 4, NQ = DIM + 2;
  __shared__ __align__(16) float s_v[64];  // chunk_velocities reads groups of 4
  __shared__ float2 s_tot[MOM_WARPS * MOM_GP][NQ];
  for (int t = threadIdx.x; t < cv.nv; t += blockDim.x) s_v[t] = cv.vnodes_f[t];
  __syncthreads();
  const int W = blockDim.x >> 5, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b0 = blockIdx.x * W * gp, i0 = b0 + warp * gp;
  const int np = min(gp, cv.n - i0);  // (none or negative in the last CTA's idle warps)
  const int nv = cv.nv, NV = cv.NV, NVp = cv.NVp;
  const int vk0 = SH ? cv.vk0 : 0;
  const float inv_nv = 1.0f / (float)nv;
  for (int g = 0; g < np; ++g) {
    const S* fi = f + (int64_t)(i0 + g) * NC * NVp;
    float msum[NQ], mcmp[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) { msum[q] = 0.0f; mcmp[q] = 0.0f; }
#pragma unroll 8
    for (int chunk = lane; chunk * VPL < NVp; chunk += 32) {
      const int k0 = chunk * VPL;
      float vel[VPL][DIM];
      bool kin[VPL];
      chunk_velocities<DIM, VPL, ROW>(k0 + vk0, nv, NV + vk0, inv_nv, s_v, vel, kin);
      float gv[NC][VPL];
#pragma unroll
      for (int c = 0; c < NC; ++c) ldv<S, VPL>(fi + (int64_t)c * NVp + k0, gv[c]);
      float ps[NQ];
#pragma unroll
      for (int q = 0; q < NQ; ++q) ps[q] = 0.0f;
#pragma unroll
      for (int e = 0; e < VPL; ++e) {
        const float g0 = kin[e] ? gv[0][e] : 0.0f;
        float v2 = 0.0f;
        ps[0] += g0;
#pragma unroll
        for (int a = 0; a < DIM; ++a) { ps[1 + a] = fmaf(vel[e][a], g0, ps[1 + a]); v2 = fmaf(vel[e][a], vel[e][a], v2); }
        ps[DIM + 1] = fmaf(v2, g0, ps[DIM + 1]);
        if (NC == 2) ps[DIM + 1] += kin[e] ? gv[NC - 1][e] : 0.0f;
      }
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        const float y = ps[q] - mcmp[q];
        const float t = msum[q] + y;
        mcmp[q] = (t - msum[q]) - y;
        msum[q] = t;
      }
    }
    // warp totals as FP32 pairs (every lane ends with the same pair)
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      float hi = msum[q], lo = -mcmp[q];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
        pair_add(hi, lo, __shfl_xor_sync(0xffffffffu, hi, o), __shfl_xor_sync(0xffffffffu, lo, o));
      if (lane == 0) s_tot[warp * gp + g][q] = make_float2(hi, lo);
    }
  }
  __syncthreads();
  const int i = b0 + threadIdx.x;
  if (threadIdx.x >= W * gp || i >= cv.n) return;
  double tot[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) tot[q] = (double)s_tot[threadIdx.x][q].x + (double)s_tot[threadIdx.x][q].y;
  if (SH) {
#pragma unroll
    for (int q = 0; q < NQ; ++q) cv.xs[(int64_t)i * NQ + q] = tot[q];
  } else {
    double rho, Un[3] = {0, 0, 0}, T;
    const double wv = cv.wv;
    finish_moments<DIM>(tot, wv, &rho, Un, &T);
    double* mo = cv.mom + (int64_t)i * MOM_STRIDE;
    mo[0] = rho; mo[1] = Un[0]; mo[2] = Un[1]; mo[3] = Un[2]; mo[4] = T;
  }
}

int launch_moments(const CaseView& cv, const void* f, cudaStream_t s) {
  const int gp = moments_gp(cv.n), W = moments_warps(cv.n), grid = (cv.n + W * gp - 1) / (W * gp);
  const bool row = cv.nv % 4 == 0;
#define BGK_MOM_WP(S, D)                                                                               \
  {                                                                                                    \
    if (row) k_moments_wp<S, D, true><<<grid, 32 * W, 0, s>>>(cv, (const S*)f, gp);                    \
    else k_moments_wp<S, D, false><<<grid, 32 * W, 0, s>>>(cv, (const S*)f, gp);                       \
  }
  if (cv.dim == 2) {
    if (cv.storage == 0) k_moments<double, double, 2><<<cv.n, 256, 0, s>>>(cv, (const double*)f);
    else if (cv.storage == 1) BGK_MOM_WP(float, 2)
    else BGK_MOM_WP(__nv_bfloat16, 2)
  } else {
    if (cv.storage == 0) k_moments<double, double, 3><<<cv.n, 256, 0, s>>>(cv, (const double*)f);
    else if (cv.storage == 1) BGK_MOM_WP(float, 3)
    else BGK_MOM_WP(__nv_bfloat16, 3)
  }
#undef BGK_MOM_WP
  return 1;
}

// ---------------------------------------------------------------------------
// velocity-sharded step: slabs of the velocity grid, each advanced by the kernels
// above with its velocity offset; the slabs couple only through the sums in cv.xs
// ---------------------------------------------------------------------------
template <typename S, int DIM>
static void launch_shard_transport_wp(const CaseView& cv, cudaStream_t s) {
  const int W = BGK_WP_WARPS, threads = 32 * W;
  const size_t smem = wp_smem_bytes<DIM>(W, cv.cap);
  const int grid = (cv.n_int + W - 1) / W;
  const bool row4 = cv.nv % 4 == 0;
#define BGK_LAUNCH_SH(ALE, ROW)                                                           \
  {                                                                                       \
    auto k = k_transport_wp<S, DIM, ALE, ROW, 4, true>;                                   \
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);       \
    k<<<grid, threads, smem, s>>>(cv);                                                    \
  }
  if (cv.ale) {
    if (row4) BGK_LAUNCH_SH(true, true) else BGK_LAUNCH_SH(true, false)
  } else {
    if (row4) BGK_LAUNCH_SH(false, true) else BGK_LAUNCH_SH(false, false)
  }
#undef BGK_LAUNCH_SH
}

int launch_shard_transport(const CaseView& cv, cudaStream_t s) {
  if (cv.n_int == 0) return 0;
  if (cv.storage == 0) return launch_transport_f64_shard(cv, s);
  if (cv.dim == 2) {
    if (cv.storage == 1) launch_shard_transport_wp<float, 2>(cv, s);
    else launch_shard_transport_wp<__nv_bfloat16, 2>(cv, s);
  } else {
    if (cv.storage == 1) launch_shard_transport_wp<float, 3>(cv, s);
    else launch_shard_transport_wp<__nv_bfloat16, 3>(cv, s);
  }
  return 1;
}

template <typename S, int DIM>
static void launch_shard_relax_wp(const CaseView& cv, cudaStream_t s) {
  const int W = 8, grid = (cv.n_int + W - 1) / W;
  if (cv.nv % 4 == 0) k_shard_relax_wp<S, DIM, true><<<grid, 32 * W, 0, s>>>(cv);
  else k_shard_relax_wp<S, DIM, false><<<grid, 32 * W, 0, s>>>(cv);
}

int launch_shard_relax(const CaseView& cv, cudaStream_t s) {
  if (cv.n_int == 0) return 0;
  if (cv.storage == 0) return launch_shard_relax_f64(cv, s);
  if (cv.dim == 2) {
    if (cv.storage == 1) launch_shard_relax_wp<float, 2>(cv, s);
    else launch_shard_relax_wp<__nv_bfloat16, 2>(cv, s);
  } else {
    if (cv.storage == 1) launch_shard_relax_wp<float, 3>(cv, s);
    else launch_shard_relax_wp<__nv_bfloat16, 3>(cv, s);
  }
  return 1;
}

int launch_shard_walls(const CaseView& cv, int phase, cudaStream_t s) {
  if (cv.n_wall == 0) return 0;
  const size_t smem = RED_BYTES + NODE_BYTES + align16(sizeof(int32_t) * (cv.cap + 1)) + sizeof(double) * cv.cap;
#define BGK_WALLS_PH(S, C, D)                                                          \
  {                                                                                    \
    if (phase == 1) k_walls<S, C, D, 1><<<cv.n_wall, 256, smem, s>>>(cv);              \
    else k_walls<S, C, D, 2><<<cv.n_wall, 256, smem, s>>>(cv);                         \
  }
  if (cv.dim == 2) {
    if (cv.storage == 0) BGK_WALLS_PH(double, double, 2)
    else if (cv.storage == 1) BGK_WALLS_PH(float, float, 2)
    else BGK_WALLS_PH(__nv_bfloat16, float, 2)
  } else {
    if (cv.storage == 0) BGK_WALLS_PH(double, double, 3)
    else if (cv.storage == 1) BGK_WALLS_PH(float, float, 3)
    else BGK_WALLS_PH(__nv_bfloat16, float, 3)
  }
#undef BGK_WALLS_PH
  return 1;
}

int launch_shard_partial(const CaseView& cv, cudaStream_t s) {
  const int gp = moments_gp(cv.n), W = moments_warps(cv.n), grid = (cv.n + W * gp - 1) / (W * gp);
  const bool row = cv.nv % 4 == 0;
#define BGK_PART_WP(S, D)                                                                                   \
  {                                                                                                         \
    if (row) k_moments_wp<S, D, true, true><<<grid, 32 * W, 0, s>>>(cv, (const S*)cv.f_in, gp);             \
    else k_moments_wp<S, D, false, true><<<grid, 32 * W, 0, s>>>(cv, (const S*)cv.f_in, gp);                \
  }
  if (cv.dim == 2) {
    if (cv.storage == 0) k_moments<double, double, 2, true><<<cv.n, 256, 0, s>>>(cv, (const double*)cv.f_in);
    else if (cv.storage == 1) BGK_PART_WP(float, 2)
    else BGK_PART_WP(__nv_bfloat16, 2)
  } else {
    if (cv.storage == 0) k_moments<double, double, 3, true><<<cv.n, 256, 0, s>>>(cv, (const double*)cv.f_in);
    else if (cv.storage == 1) BGK_PART_WP(float, 3)
    else BGK_PART_WP(__nv_bfloat16, 3)
  }
#undef BGK_PART_WP
  return 1;
}

template <int DIM>
__global__ void k_shard_moments(CaseView cv) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= cv.n) return;
  double tot[DIM + 2];
#pragma unroll
  for (int q = 0; q < DIM + 2; ++q) tot[q] = cv.xs[(int64_t)i * (DIM + 2) + q];
  double rho, Un[3] = {0, 0, 0}, T;
  const double wv = cv.wv;
  finish_moments<DIM>(tot, wv, &rho, Un, &T);
  double* mo = cv.mom + (int64_t)i * MOM_STRIDE;
  mo[0] = rho; mo[1] = Un[0]; mo[2] = Un[1]; mo[3] = Un[2]; mo[4] = T;
}

int launch_shard_moments(const CaseView& cv, cudaStream_t s) {
  if (cv.dim == 2) k_shard_moments<2><<<grid_for(cv.n, 256), 256, 0, s>>>(cv);
  else k_shard_moments<3><<<grid_for(cv.n, 256), 256, 0, s>>>(cv);
  return 1;
}

// One-device stand-in for the allreduce of the slabs' sums: every element is summed
// over the buffers in buffer order and the sum is written to every buffer, so that
// all slabs continue from the same bits.
struct ShardBufs {
  double* p[SHARD_MAX_BUFS];
};

__global__ void k_shard_allreduce(ShardBufs b, int nb, int64_t count) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < count; e += (int64_t)gridDim.x * blockDim.x) {
    double sum = 0.0;
    for (int r = 0; r < nb; ++r) sum += b.p[r][e];
    for (int r = 0; r < nb; ++r) b.p[r][e] = sum;
  }
}

int launch_shard_allreduce(double* const* bufs, int nbufs, int64_t count, cudaStream_t s) {
  if (count <= 0) return 0;
  ShardBufs b;
  for (int r = 0; r < SHARD_MAX_BUFS; ++r) b.p[r] = r < nbufs ? bufs[r] : nullptr;
  const int64_t blocks = (count + 255) / 256;
  k_shard_allreduce<<<(int)(blocks < 4096 ? blocks : 4096), 256, 0, s>>>(b, nbufs, count);
  return 1;
}

// Copies between the caller's dense layout and the padded storage, converting the element
// type.  Both are bound by HBM.
//   Without padding (NV % 4 == 0) the arrays are flat: 4 elements per thread and access, four
// accesses in flight (16-byte loads and stores in FP32; pointers aligned to 4 elements):
// 101^2 x 24^2 FP32 (94 MB) 11 us, 33 us with one element per thread and a 64-bit division.
//   Rows of 256 elements and more: a warp takes whole rows, so that every access of 32
// neighbouring elements is contiguous whatever the row's alignment, eight of them in flight
// and no thread divides: 133^2 x 27^2 FP32 (206 MB) 40 us, 82 us by elements with a division.
//   Shorter rows leave a warp fewer than eight accesses: a CTA takes the elements of a block
// of whole destination rows in turn and steps through them by additions: 301^2 x 13^2 39 us
// (69 us by rows), 201^2 x 5^2 7 us (9 us).  Elements past the end load the first one, so
// that no load waits for a branch.
template <typename A, typename B>
__global__ void __launch_bounds__(256) k_convert_flat(const A* __restrict__ src, B* __restrict__ dst, int64_t n4) {
  using CA = decltype(ld1(src));
  using CB = decltype(ld1(dst));
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n4; t += 4 * stride) {
    CA v[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (t + u * stride < n4) ld4(src + 4 * (t + u * stride), v[u]);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (t + u * stride < n4) {
        const CB w[4] = {(CB)v[u][0], (CB)v[u][1], (CB)v[u][2], (CB)v[u][3]};
        st4(dst + 4 * (t + u * stride), w);
      }
  }
}

template <typename A, typename B>
__global__ void __launch_bounds__(256) k_convert_rows(const A* __restrict__ src, B* __restrict__ dst, int64_t rows,
                                                      int NV, int ls, int ld) {
  using CB = decltype(ld1(dst));
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int64_t r = (int64_t)blockIdx.x * nw + (threadIdx.x >> 5); r < rows; r += (int64_t)gridDim.x * nw) {
    const A* a = src + r * ls;
    B* b = dst + r * ld;
#pragma unroll 8
    for (int k = lane; k < ld; k += 32) st1(b + k, k < NV ? (CB)ld1(a + k) : (CB)0);
  }
}

constexpr int kShortRow = 256;       // elements of a row from which it is copied by a warp
constexpr int kConvertTile = 4096;   // elements of a block of shorter rows
template <typename A, typename B, bool PAD>
__global__ void __launch_bounds__(256) k_convert_short(const A* __restrict__ src, B* __restrict__ dst, int64_t rows,
                                                      int NV, int ls, int ld, int per, int dk, int dsrc) {
  using CB = decltype(ld1(dst));
  const int64_t r0 = (int64_t)blockIdx.x * per;
  const int m = (int)min((int64_t)per, rows - r0) * ld;
  const int q = fdiv_small(threadIdx.x, 1.0f / (float)ld);
  int k = threadIdx.x - q * ld;  // position in the row
  const A* a = src + r0 * ls + q * ls + k;
  B* b = dst + r0 * ld + threadIdx.x;
  for (int t = threadIdx.x; t < m; t += 8 * 256, b += 8 * 256) {
    CB v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const bool on = t + u * 256 < m && (!PAD || k < NV);
      v[u] = (CB)ld1(on ? a : src);
      if (PAD && !on) v[u] = (CB)0;
      k += dk;
      a += dsrc;
      if (k >= ld) { k -= ld; a += ls - ld; }
    }
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (t + u * 256 < m) st1(b + u * 256, v[u]);
  }
}

template <typename A, typename B>
static void convert(const A* src, B* dst, int64_t rows, int NV, int ls, int ld, cudaStream_t s) {
  if (ls == ld && NV == ls && reinterpret_cast<uintptr_t>(src) % (4 * sizeof(A) < 16 ? 4 * sizeof(A) : 16) == 0 &&
      reinterpret_cast<uintptr_t>(dst) % (4 * sizeof(B) < 16 ? 4 * sizeof(B) : 16) == 0) {
    const int64_t n4 = rows * ls / 4;  // (NV is a multiple of 4 here: ls = ld = NV is the padded length)
    k_convert_flat<<<(int)std::min<int64_t>((n4 + 1023) / 1024, TARGET_SMS * 32), 256, 0, s>>>(src, dst, n4);
  } else if (ld >= kShortRow) {
    k_convert_rows<<<(int)std::min<int64_t>((rows + 7) / 8, TARGET_SMS * 64), 256, 0, s>>>(src, dst, rows, NV, ls, ld);
  } else {
    // a step of 256 elements: 256 / ld rows and dk elements on (one row more where dk wraps)
    const int per = kConvertTile / ld, dk = 256 % ld, dsrc = 256 / ld * ls + dk;
    const int grid = (int)((rows + per - 1) / per);
    if (ld > NV) k_convert_short<A, B, true><<<grid, 256, 0, s>>>(src, dst, rows, NV, ls, ld, per, dk, dsrc);
    else k_convert_short<A, B, false><<<grid, 256, 0, s>>>(src, dst, rows, NV, ls, ld, per, dk, dsrc);
  }
}

template <typename A>
static void pack_from(const CaseView& cv, const A* src, void* dst, cudaStream_t s) {
  const int64_t rows = (int64_t)cv.n * cv.ncomp;
  if (cv.storage == 0) convert(src, (double*)dst, rows, cv.NV, cv.NV, cv.NVp, s);
  else if (cv.storage == 1) convert(src, (float*)dst, rows, cv.NV, cv.NV, cv.NVp, s);
  else convert(src, (__nv_bfloat16*)dst, rows, cv.NV, cv.NV, cv.NVp, s);
}

template <typename B>
static void unpack_to(const CaseView& cv, const void* src, B* dst, cudaStream_t s) {
  const int64_t rows = (int64_t)cv.n * cv.ncomp;
  if (cv.storage == 0) convert((const double*)src, dst, rows, cv.NV, cv.NVp, cv.NV, s);
  else if (cv.storage == 1) convert((const float*)src, dst, rows, cv.NV, cv.NVp, cv.NV, s);
  else convert((const __nv_bfloat16*)src, dst, rows, cv.NV, cv.NVp, cv.NV, s);
}

int launch_pack_f(const CaseView& cv, const void* src, int src_dtype, void* dst, cudaStream_t s) {
  if (src_dtype == 0) pack_from(cv, (const double*)src, dst, s);
  else if (src_dtype == 1) pack_from(cv, (const float*)src, dst, s);
  else pack_from(cv, (const __nv_bfloat16*)src, dst, s);
  return 1;
}

int launch_unpack_f(const CaseView& cv, const void* src, void* dst, int dst_dtype, cudaStream_t s) {
  if (dst_dtype == 0) unpack_to(cv, src, (double*)dst, s);
  else if (dst_dtype == 1) unpack_to(cv, src, (float*)dst, s);
  else unpack_to(cv, src, (__nv_bfloat16*)dst, s);
  return 1;
}

}  // namespace bgk
