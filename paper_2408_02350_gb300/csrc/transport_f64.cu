// Transport, moments and relaxation with FP64 storage (Sec. 3.2, 3.4.2), and the
// relaxations of the second-order and velocity-sharded steps on FP64 rows.
//
// Bound: the FP64 pipe.  FP64 runs at 2 lanes per clock per SM on GB300 (0.62 T FMA/s
// measured), so a warp instruction in FP64 holds the pipe for 16 cycles and everything
// else (integer selects, loads, issue slots) is nearly free beside it.  The kernel is
// therefore written for few FP64 instructions per (point, neighbour, velocity):
//   - a thread's 4 consecutive velocities lie in one row of the velocity grid (ROW,
//     nv % 4 == 0), so c.P_d is one FMA from a base shared by the row;
//   - min(c.P_d, 0) is an integer test of the sign (min_zero), not an FP64 comparison;
//   - fixed points (MIR): v and its mirror -v share their projections, since the sign
//     splits p_d into min(p_d, 0) and max(p_d, 0) = -min(-p_d, 0), both exact: 5.3
//     FP64 instructions per (point, neighbour, velocity) in 2D instead of 6.5, and 11
//     with neither;
//   - the Maxwellian is a product of one exponential per axis and grid node (nv DIM
//     exponentials per point instead of nv^DIM), the moments come from row sums, and
//     the four moment sums are reduced across the warp transposed.
// f~ goes to the output row and is read back from there for the relaxation, so a thread
// takes any number of velocity chunks.
// 41^2 points x 16^2 velocities, fixed points: 104 us per launch with the FP64 pipe 84 %
// busy (221 us with c.P_d in full per velocity, FP64 comparisons and one exponential per
// velocity).
#include <algorithm>

#include "bgk_internal.cuh"
#include "device_common.cuh"

namespace bgk {

namespace {

constexpr int kWarpsMax = 8;
constexpr int kAxis = 64;  // most nodes per axis

// min(p, 0) and max(p, 0) by the sign bit (NaN gives 0, as fmin(NaN, 0) and fmax do).
__device__ __forceinline__ double min_zero(double p) {
  const uint32_t hi = (uint32_t)__double2hiint(p);
  return hi - 0x80000000u <= 0x7ff00000u ? p : 0.0;
}
__device__ __forceinline__ double max_zero(double p) {
  const uint32_t hi = (uint32_t)__double2hiint(p);
  return hi <= 0x7ff00000u ? p : 0.0;
}

// Shared memory: velocity nodes and their squares, the axis exponentials, the warps'
// moment sums, the broadcast results; the list and the stencil of the point follow.
struct F64Shared {
  double v[kAxis], v2[kAxis], ex[3 * kAxis];
  double sum[kWarpsMax][8];
  double fin[8];
};

inline size_t f64_smem(int cap, int dd) {
  return sizeof(F64Shared) + ((sizeof(int32_t) * cap + 15) & ~size_t(15)) + sizeof(double) * (size_t)cap * dd;
}

// First component index and the rows (other axes) of the 4 velocities from flattened grid
// index k: with ROW they share iy, iz.
template <int DIM, bool ROW>
__device__ __forceinline__ void split4(int k, int nv, int last, int (&ia)[4][DIM]) {
  if (ROW) {
    int q = k / nv;
    const int x0 = k - q * nv;
#pragma unroll
    for (int e = 0; e < 4; ++e) ia[e][0] = x0 + e;
#pragma unroll
    for (int a = 1; a < DIM; ++a) {
      const int r = q / nv;
#pragma unroll
      for (int e = 0; e < 4; ++e) ia[e][a] = q - r * nv;
      q = r;
    }
  } else {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      int kk = k + e < last ? k + e : 0;
#pragma unroll
      for (int a = 0; a < DIM; ++a) {
        const int q = kk / nv;
        ia[e][a] = kk - q * nv;
        kk = q;
      }
    }
  }
}

// Moment sums of 4 velocities: R += g, M_a += v_a g, E += |v|^2 g (+ h).
template <int DIM, bool ROW>
__device__ __forceinline__ void add_moments(const F64Shared& sm, const int (&ia)[4][DIM], const double (&ft)[2][4],
                                            int nin, double (&part)[DIM + 2]) {
  if (ROW && nin == 4) {
    double r = 0.0, x = 0.0, e2 = 0.0;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const double g = ft[0][e];
      r += g;
      x = fma(sm.v[ia[e][0]], g, x);
      e2 = fma(sm.v2[ia[e][0]], g, e2);
      if (DIM == 2) e2 += ft[1][e];
    }
    part[0] += r;
    part[1] += x;
#pragma unroll
    for (int a = 1; a < DIM; ++a) {
      part[1 + a] = fma(sm.v[ia[0][a]], r, part[1 + a]);
      e2 = fma(sm.v2[ia[0][a]], r, e2);
    }
    part[DIM + 1] += e2;
  } else {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      if (e >= nin) continue;
      const double g = ft[0][e];
      part[0] += g;
#pragma unroll
      for (int a = 0; a < DIM; ++a) {
        part[1 + a] = fma(sm.v[ia[e][a]], g, part[1 + a]);
        part[DIM + 1] = fma(sm.v2[ia[e][a]], g, part[DIM + 1]);
      }
      if (DIM == 2) part[DIM + 1] += ft[1][e];
    }
  }
}

// Totals of the threads' sums over the CTA; every thread gets them.  Within a warp four
// sums are reduced transposed (2 + 1 + 3 additions instead of 4 x 5).
template <int N>
__device__ __forceinline__ void cta_totals(F64Shared& sm, double (&s)[N], double (&tot)[N]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const bool h16 = (lane & 16) != 0, h8 = (lane & 8) != 0;
  double a = h16 ? s[2] : s[0], b = h16 ? s[3] : s[1];
  a += __shfl_xor_sync(0xffffffffu, h16 ? s[0] : s[2], 16);
  b += __shfl_xor_sync(0xffffffffu, h16 ? s[1] : s[3], 16);
  double k = h8 ? b : a;
  k += __shfl_xor_sync(0xffffffffu, h8 ? a : b, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
  if ((lane & 7) == 0) sm.sum[warp][lane >> 3] = k;
#pragma unroll
  for (int q = 4; q < N; ++q) {
    const double t = warp_sum(s[q]);
    if (lane == 0) sm.sum[warp][q] = t;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < N; ++q) {
    double t = sm.sum[0][q];
    for (int w = 1; w < nw; ++w) t += sm.sum[w][q];
    tot[q] = t;
  }
}

// Moments from the raw sums, tau and the relaxation of the output row (which holds f~):
// f^{n+1} = (tau f~ + dt M)/(tau + dt), or with RK = 1 the exact relaxation over dt/2.
// The lanes of the first warp form the moments, each the same (the FP64 pipe works per warp,
// so one lane would cost the same).  The row starts at grid velocity vk0.
template <int DIM, bool ROW, int RK>
__device__ __forceinline__ void relax_f64(const CaseView& cv, F64Shared& sm, const int i, const double (&tot)[DIM + 2],
                                          const int vk0) {
  constexpr int NC = DIM == 2 ? 2 : 1;
  const int nv = cv.nv, NV = cv.NV, NVp = cv.NVp, nchunk = NVp >> 2;
  if (threadIdx.x < 32) {
    const double R = tot[0], rR = 1.0 / R;
    double U[DIM], u2 = 0.0;
#pragma unroll
    for (int a = 0; a < DIM; ++a) { U[a] = tot[1 + a] * rR; u2 = fma(U[a], U[a], u2); }
    const double T = fma(-R, u2, tot[DIM + 1]) * rR / 3.0, rho = R * cv.wv;
    const bool bad = !(rho > 0.0) || !(T > 0.0) || !isfinite(rho) || !isfinite(T);
    double a = 1.0, bp = 0.0, i2T = 0.0;
    if (!bad && cv.tau_mode != 2) {
      const double pi = 3.14159265358979323846, sq = 0.79788456080286535588;  // sqrt(2 / pi)
      const double tau = cv.tau_mode == 1 ? sq * cv.kn : sq * cv.kn / (rho * sqrt(T));
      double b;
      if (RK == 1) {
        a = exp(-0.5 * cv.dt / tau);
        b = -expm1(-0.5 * cv.dt / tau);
      } else {
        const double q = 1.0 / (tau + cv.dt);
        a = tau * q;
        b = cv.dt * q;
      }
      i2T = 0.5 / T;
      const double z = i2T / pi;  // 1 / (2 pi T)
      bp = b * rho * z * (DIM == 2 ? 1.0 : sqrt(z));
    }
    if (threadIdx.x == 0) {
      double* mo = cv.mom + (int64_t)i * MOM_STRIDE;
      mo[0] = rho;
#pragma unroll
      for (int q = 0; q < 3; ++q) mo[1 + q] = q < DIM ? U[q < DIM ? q : 0] : 0.0;
      mo[4] = T;
      if (bad) set_status(cv.status, ST_NONFINITE);
      sm.fin[0] = a; sm.fin[1] = bp; sm.fin[2] = i2T; sm.fin[3] = T;
#pragma unroll
      for (int q = 0; q < DIM; ++q) sm.fin[4 + q] = U[q];
    }
  }
  __syncthreads();
  const double ca = sm.fin[0], T = sm.fin[3];
  // exponentials per axis and node, the prefactor in the first axis
  for (int t = threadIdx.x; t < DIM * nv; t += blockDim.x) {
    const int a = t / nv, j = t - a * nv;
    const double d = sm.v[j] - sm.fin[4 + a];
    const double x = exp(-d * d * sm.fin[2]);
    sm.ex[a * kAxis + j] = a == 0 ? sm.fin[1] * x : x;
  }
  __syncthreads();
  double* fo = reinterpret_cast<double*>(cv.f_out) + (int64_t)i * NC * NVp;
  for (int chunk = threadIdx.x; chunk < nchunk; chunk += blockDim.x) {
    const int k0 = 4 * chunk;
    int ia[4][DIM];
    split4<DIM, ROW>(k0 + vk0, nv, NV + vk0, ia);
    double f[NC][4];
#pragma unroll
    for (int c = 0; c < NC; ++c) ld4(fo + (int64_t)c * NVp + k0, f[c]);
    double base = 1.0;
    if (ROW) {
      base = sm.ex[kAxis + ia[0][1]];
      if (DIM == 3) base *= sm.ex[2 * kAxis + ia[0][DIM - 1]];
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      double M = sm.ex[ia[e][0]];
      if (ROW) {
        M *= base;
      } else {
#pragma unroll
        for (int a = 1; a < DIM; ++a) M *= sm.ex[a * kAxis + ia[e][a]];
      }
      const bool in = k0 + e < NV;
      f[0][e] = in ? fma(ca, f[0][e], M) : 0.0;
      if (NC == 2) f[NC - 1][e] = in ? fma(ca, f[NC - 1][e], T * M) : 0.0;
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) st4(fo + (int64_t)c * NVp + k0, f[c]);
  }
}

__device__ __forceinline__ void load_nodes(const CaseView& cv, F64Shared& sm) {
  for (int t = threadIdx.x; t < cv.nv; t += blockDim.x) {
    const double v = cv.vnodes[t];
    sm.v[t] = v;
    sm.v2[t] = v * v;
  }
}

// f~ = f_i - 2 dt (acc - sk f_i) of one chunk (averaged with the step's starting row when
// AVG), written to the output row and added to the moment sums.
template <int DIM, bool ROW, bool AVG>
__device__ __forceinline__ void chunk_out(const CaseView& cv, const F64Shared& sm, const int i, const int k0,
                                          const int (&ia)[4][DIM], const double (&acc)[2][4], const double (&sk)[4],
                                          const double two_dt, double (&part)[DIM + 2]) {
  constexpr int NC = DIM == 2 ? 2 : 1;
  const int NVp = cv.NVp;
  const int64_t o = (int64_t)i * NC * NVp + k0;
  const double* fi = reinterpret_cast<const double*>(cv.f_in) + o;
  double* fo = reinterpret_cast<double*>(cv.f_out) + o;
  const int nin = min(4, cv.NV - k0);
  double ft[2][4];
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    double f[4];
    ld4(fi + (int64_t)c * NVp, f);
#pragma unroll
    for (int e = 0; e < 4; ++e) ft[c][e] = fma(-two_dt, fma(-sk[e], f[e], acc[c][e]), f[e]);
    if (AVG) {
      double fa[4];
      ld4(reinterpret_cast<const double*>(cv.f_avg) + o + (int64_t)c * NVp, fa);
#pragma unroll
      for (int e = 0; e < 4; ++e) ft[c][e] = 0.5 * (ft[c][e] + fa[e]);
    }
  }
  add_moments<DIM, ROW>(sm, ia, ft, nin, part);
#pragma unroll
  for (int c = 0; c < NC; ++c) {
#pragma unroll
    for (int e = 0; e < 4; ++e) ft[c][e] = e < nin ? ft[c][e] : 0.0;
    st4(fo + (int64_t)c * NVp, ft[c]);
  }
}

// One CTA per interior point, a thread per chunk of 4 velocities (MIR: per chunk of the
// first half of the grid and its mirror).  SH: the raw moment sums of the velocity slab to
// the exchange buffer instead of the relaxation.  AVG: the second stage of the
// second-order step.
template <int DIM, bool ROW, bool ALE, bool SH, bool AVG, bool MIR>
__global__ void __launch_bounds__(32 * kWarpsMax) k_transport_f64(const CaseView cv) {
  constexpr int NC = DIM == 2 ? 2 : 1, DD = DIM * DIM;
  extern __shared__ __align__(16) unsigned char smem[];
  F64Shared& sm = *reinterpret_cast<F64Shared*>(smem);
  int32_t* s_col = reinterpret_cast<int32_t*>(smem + sizeof(F64Shared));
  double* s_P = reinterpret_cast<double*>(smem + sizeof(F64Shared) + ((sizeof(int32_t) * cv.cap + 15) & ~size_t(15)));
  const int i = cv.int_idx[blockIdx.x];
  const int m = checked_count(cv.cnt[i], cv.cap, cv.status);
  const int nv = cv.nv, NV = cv.NV, NVp = cv.NVp;
  const int vk0 = SH ? cv.vk0 : 0;
  load_nodes(cv, sm);
  {
    const int32_t* col = cv.col + (int64_t)i * cv.cap;
    const double* P = reinterpret_cast<const double*>(cv.P) + (int64_t)i * cv.cap * DD;
    for (int t = threadIdx.x; t < m; t += blockDim.x) s_col[t] = checked_index(col[t], cv.n, i, cv.status);
    for (int t = threadIdx.x; t < m * DD; t += blockDim.x) s_P[t] = P[t];
  }
  __syncthreads();
  double U[DIM];
#pragma unroll
  for (int a = 0; a < DIM; ++a) U[a] = ALE ? cv.mom[(int64_t)i * MOM_STRIDE + 1 + a] : 0.0;
  const double* fbase = reinterpret_cast<const double*>(cv.f_in);
  const int64_t rowlen = (int64_t)NC * NVp;
  const double two_dt = 2.0 * cv.dt;
  double part[DIM + 2];
#pragma unroll
  for (int t = 0; t < DIM + 2; ++t) part[t] = 0.0;
  const int nchunk = MIR ? NV / 8 : NVp >> 2;
  for (int chunk = threadIdx.x; chunk < nchunk; chunk += blockDim.x) {
    const int k0 = 4 * chunk, km = NV - 4 - k0;
    int ia[4][DIM];
    split4<DIM, ROW>(k0 + vk0, nv, NV + vk0, ia);
    double c[4][DIM];
#pragma unroll
    for (int e = 0; e < 4; ++e)
#pragma unroll
      for (int a = 0; a < DIM; ++a)
        if (!ROW || a == 0 || e == 0) c[e][a] = sm.v[ia[e][a]] - U[a];
    double acc[2][4], sk[4], accm[2][4], skm[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      sk[e] = 0.0;
      skm[e] = 0.0;
#pragma unroll
      for (int q = 0; q < 2; ++q) { acc[q][e] = 0.0; accm[q][e] = 0.0; }
    }
    const double* f0 = fbase + k0;
    const double* f1 = fbase + km;
    for (int s = 0; s < m; ++s) {
      const int64_t o = (int64_t)s_col[s] * rowlen;
      double f[NC][4], fm[NC][4];
#pragma unroll
      for (int q = 0; q < NC; ++q) {
        ld4(f0 + o + (int64_t)q * NVp, f[q]);
        if (MIR) ld4(f1 + o + (int64_t)q * NVp, fm[q]);
      }
      double mk[4], qk[4];
#pragma unroll
      for (int d = 0; d < DIM; ++d) {
        const double* P = s_P + s * DD + d * DIM;
        double b = 0.0;
        if (ROW) {
          b = c[0][1] * P[1];
          if (DIM == 3) b = fma(c[0][DIM - 1], P[DIM - 1], b);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (!ROW) {
            b = c[e][1] * P[1];
            if (DIM == 3) b = fma(c[e][DIM - 1], P[DIM - 1], b);
          }
          const double p = fma(c[e][0], P[0], b);
          const double lo = min_zero(p);
          mk[e] = d == 0 ? lo : mk[e] + lo;
          if (MIR) {
            const double hi = max_zero(p);
            qk[e] = d == 0 ? hi : qk[e] + hi;
          }
        }
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        sk[e] += mk[e];
#pragma unroll
        for (int q = 0; q < NC; ++q) acc[q][e] = fma(mk[e], f[q][e], acc[q][e]);
        if (MIR) {
          // m(-v) = -qk; element 3 - e of the mirror chunk holds -v_e
          skm[3 - e] -= qk[e];
#pragma unroll
          for (int q = 0; q < NC; ++q) accm[q][3 - e] = fma(-qk[e], fm[q][3 - e], accm[q][3 - e]);
        }
      }
    }
    chunk_out<DIM, ROW, AVG>(cv, sm, i, k0, ia, acc, sk, two_dt, part);
    if (MIR) {
      int ib[4][DIM];
#pragma unroll
      for (int e = 0; e < 4; ++e)
#pragma unroll
        for (int a = 0; a < DIM; ++a) ib[e][a] = nv - 1 - ia[3 - e][a];
      chunk_out<DIM, ROW, AVG>(cv, sm, i, km, ib, accm, skm, two_dt, part);
    }
  }
  double tot[DIM + 2];
  cta_totals<DIM + 2>(sm, part, tot);
  if constexpr (SH) {
    if (threadIdx.x == 0) {
#pragma unroll
      for (int q = 0; q < DIM + 2; ++q) cv.xs[(int64_t)i * (DIM + 2) + q] = tot[q];
    }
  } else {
    relax_f64<DIM, ROW, AVG ? 1 : 0>(cv, sm, i, tot, 0);
  }
}

// Relaxation of the output rows in place.  SH (sharded step): with the moments of the
// summed sums in the exchange buffer; else (second-order step): the exact relaxation over
// dt/2 with the row's own moments.
template <int DIM, bool ROW, bool SH>
__global__ void __launch_bounds__(32 * kWarpsMax) k_relax_f64(const CaseView cv) {
  constexpr int NC = DIM == 2 ? 2 : 1;
  __shared__ F64Shared sm;
  const int i = cv.int_idx[blockIdx.x];
  const int NVp = cv.NVp, nchunk = NVp >> 2;
  load_nodes(cv, sm);
  __syncthreads();
  double tot[DIM + 2];
  if constexpr (SH) {
#pragma unroll
    for (int q = 0; q < DIM + 2; ++q) tot[q] = cv.xs[(int64_t)i * (DIM + 2) + q];
    relax_f64<DIM, ROW, 0>(cv, sm, i, tot, cv.vk0);
  } else {
    const double* fo = reinterpret_cast<const double*>(cv.f_out) + (int64_t)i * NC * NVp;
    double part[DIM + 2];
#pragma unroll
    for (int t = 0; t < DIM + 2; ++t) part[t] = 0.0;
    for (int chunk = threadIdx.x; chunk < nchunk; chunk += blockDim.x) {
      int ia[4][DIM];
      split4<DIM, ROW>(4 * chunk, cv.nv, cv.NV, ia);
      double ft[2][4];
#pragma unroll
      for (int c = 0; c < NC; ++c) ld4(fo + (int64_t)c * NVp + 4 * chunk, ft[c]);
      add_moments<DIM, ROW>(sm, ia, ft, min(4, cv.NV - 4 * chunk), part);
    }
    cta_totals<DIM + 2>(sm, part, tot);
    relax_f64<DIM, ROW, 1>(cv, sm, i, tot, 0);
  }
}

int cta_threads(int nchunk) { return std::min(32 * kWarpsMax, (nchunk + 31) / 32 * 32); }

template <int DIM, bool ROW, bool SH, bool AVG>
void launch_f64(const CaseView& cv, cudaStream_t s) {
  const size_t smem = f64_smem(cv.cap, DIM * DIM);
  auto go = [&](auto k, int nchunk) {
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k<<<cv.n_int, cta_threads(nchunk), smem, s>>>(cv);
  };
  if (cv.ale && !AVG) {
    go(k_transport_f64<DIM, ROW, !AVG, SH, AVG, false>, cv.NVp / 4);
    return;
  }
  if constexpr (ROW && !SH) {
    // the whole grid in chunks of 4 that pair up: v at k, -v at NV - 1 - k (nv % 4 == 0, so
    // NV % 8 == 0)
    go(k_transport_f64<DIM, ROW, false, SH, AVG, true>, cv.NV / 8);
  } else {
    go(k_transport_f64<DIM, ROW, false, SH, AVG, false>, cv.NVp / 4);
  }
}

template <bool SH, bool AVG>
int launch_f64_any(const CaseView& cv, cudaStream_t s) {
  const bool row = cv.nv % 4 == 0;
  if (cv.dim == 2) {
    if (row) launch_f64<2, true, SH, AVG>(cv, s);
    else launch_f64<2, false, SH, AVG>(cv, s);
  } else {
    if (row) launch_f64<3, true, SH, AVG>(cv, s);
    else launch_f64<3, false, SH, AVG>(cv, s);
  }
  return 1;
}

template <bool SH>
int launch_relax_any(const CaseView& cv, cudaStream_t s) {
  const bool row = cv.nv % 4 == 0;
  const int threads = cta_threads(cv.NVp / 4);
  if (cv.dim == 2) {
    if (row) k_relax_f64<2, true, SH><<<cv.n_int, threads, 0, s>>>(cv);
    else k_relax_f64<2, false, SH><<<cv.n_int, threads, 0, s>>>(cv);
  } else {
    if (row) k_relax_f64<3, true, SH><<<cv.n_int, threads, 0, s>>>(cv);
    else k_relax_f64<3, false, SH><<<cv.n_int, threads, 0, s>>>(cv);
  }
  return 1;
}

}  // namespace

int launch_transport_f64(const CaseView& cv, cudaStream_t s) { return launch_f64_any<false, false>(cv, s); }
int launch_transport_f64_shard(const CaseView& cv, cudaStream_t s) { return launch_f64_any<true, false>(cv, s); }
int launch_transport_f64_avg(const CaseView& cv, cudaStream_t s) { return launch_f64_any<false, true>(cv, s); }
int launch_relax_half_f64(const CaseView& cv, cudaStream_t s) { return launch_relax_any<false>(cv, s); }
int launch_shard_relax_f64(const CaseView& cv, cudaStream_t s) { return launch_relax_any<true>(cv, s); }

}  // namespace bgk
