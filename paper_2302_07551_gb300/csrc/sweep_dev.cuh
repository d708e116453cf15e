// Device helpers shared by the single-chain and the batched FP64 kernels.
//
// Warp-per-level products: lane k owns rows k, k+32, ... (R = ceil(m/32)
// rows) of a column-major m x m block; input vectors sit in a per-warp
// shared-memory slice (zero beyond m) and are read as broadcast pairs.
#pragma once
#include <math.h>

#include "mc_internal.cuh"

namespace mc {
namespace dev {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ double ld_stream(const double* p) { return __ldcs(p); }

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// Warp index for the persistent loop  for (u = w; u < P; u += nw).  With
// several rounds it is block-major: a block's warps take consecutive units, so
// the grid streams one window of neighbouring levels.  When all P units fit in
// one partial round it is block-minor instead, so that the busy warps spread
// evenly over the blocks (hence over the SMs) rather than filling the first
// blocks.  Both orders are permutations of [0, nw).
__device__ __forceinline__ int sched_warp(int64_t P, int nw) {
  if (P >= nw) return (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  return (int)((threadIdx.x >> 5) * gridDim.x + blockIdx.x);
}

template <int R>
struct Tune {
  static constexpr int U = R <= 1 ? 16 : R <= 2 ? 8 : R <= 4 ? 4 : 2;  // columns per batch
  static constexpr int MINB = R <= 4 ? 3 : 2;                          // blocks per SM
};

// acc[r] += sum over columns [j0b, j1) of M(row_r, j) * v[j] of a column-major block M.
// v: shared, zero beyond m and readable to the end of the last batch (so the pair load
// at an odd end reads a zero, or meets a zero block entry).
template <int R>
__device__ __forceinline__ void gemv_acc(double (&acc)[R], const double* __restrict__ M,
                                         const double* v, int j0b, int j1, int m, int lane) {
  constexpr int U = Tune<R>::U;
  for (int j0 = j0b; j0 < j1; j0 += U) {
    double t[U][R];
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const int j = j0 + q;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int row = lane + 32 * r;
        t[q][r] = (j < j1 && row < m) ? ld_stream(M + (size_t)j * m + row) : 0.0;
      }
    }
#pragma unroll
    for (int q = 0; q < U; q += 2) {
      const double2 vv = *reinterpret_cast<const double2*>(v + j0 + q);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        acc[r] = fma(t[q][r], vv.x, acc[r]);
        acc[r] = fma(t[q + 1][r], vv.y, acc[r]);
      }
    }
  }
}

// CG: p was written by other SMs during this kernel, so it is read from L2
// (ld.global.cg), never from a possibly stale L1 line.
template <int R, bool CG = false>
__device__ __forceinline__ void stage_vec(double* v, const double* __restrict__ p, int m,
                                          int lane) {
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int row = lane + 32 * r;
    v[row] = row < m ? (CG ? __ldcg(p + row) : p[row]) : 0.0;
  }
}

template <int R>
__device__ __forceinline__ void zero_acc(double (&acc)[R]) {
#pragma unroll
  for (int r = 0; r < R; ++r) acc[r] = 0.0;
}

// Deterministic block-wide sum (fixed shuffle tree, fixed warp order).
__device__ __forceinline__ double block_sum(double v, double* sh) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) sh[w] = v;
  __syncthreads();
  double t = lane < nw ? sh[lane] : 0.0;
  t = warp_sum(t);
  return t;
}

// As block_sum, valid on thread 0 only: the second stage by one warp (every warp
// that adds costs 16 clocks of the SM's FP64 pipe per instruction).
__device__ __forceinline__ double block_sum0(double v, double* sh) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) sh[w] = v;
  __syncthreads();
  if (w == 0) {
    v = lane < nw ? sh[lane] : 0.0;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);   // nw <= 8
  }
  return v;
}

// One level of a half-sweep (Algorithm 2): z_l = (-T_dd)^{-1}(T_lo v_{l-1} +
// T_up v_{l+1}) (inverse mode: A = T_lo, B = T_up, C = (-T_dd)^{-1}) or
// z_l = W_lo v_{l-1} + W_up v_{l+1} (coupled: A = W_lo, B = W_up), written to
// dst; returns sum_i z_l[i] on every lane.  slice: 3 * 32 R doubles of the
// warp's shared memory.
// Off-staircase terms of a block-banded Q^T: acc += sum_j T_{l,l+d_j} v_{l+d_j}
// with v = xlo for d_j < 0 and xup for d_j > 0 (staged through slice).
template <int R, bool CG = false>
__device__ __forceinline__ void far_terms(double (&acc)[R], const FarDesc* far,
                                          const double* xlo, const double* xup, int64_t l,
                                          int64_t L, int m, int ms, double* slice, int lane) {
  const int n = far->n;
  for (int j = 0; j < n; ++j) {
    const int64_t k = l + far->off[j];
    if (k < 0 || k >= L) continue;
    __syncwarp();
    stage_vec<R, CG>(slice, (far->off[j] < 0 ? xlo : xup) + k * m, m, lane);
    __syncwarp();
    gemv_acc<R>(acc, far->plane[j] + (size_t)l * ms, slice, 0, m, m, lane);
  }
  __syncwarp();
}

// Returns sum_i z_l[i]: on every lane (WARP_TOTAL) or the lane's own rows
// only (callers that only need a total over many levels reduce once at the end);
// want_sum = false skips the sum (0 is returned): the FP64 adds it costs are a
// share of an FP64-bound kernel, and a fused launch only needs the sums of its
// last two sweeps.
// CG: neighbour vectors written by other SMs during this kernel (L2 reads).
template <int R, bool COUPLED, bool WARP_TOTAL = true, bool CG = false>
__device__ __forceinline__ double level_sweep2(const double* A, const double* B, const double* C,
                                               const double* src, const double* src_up,
                                               double* dst, int64_t l, int64_t L, int m, int ms,
                                               double* slice, int lane,
                                               const FarDesc* far = nullptr,
                                               const double* xfar_lo = nullptr,
                                               const double* xfar_up = nullptr,
                                               bool want_sum = true) {
  constexpr int W = 32 * R;
  double* v_lo = slice;
  double* v_up = slice + W;
  double* v_g = slice + 2 * W;
  const bool has_lo = l > 0, has_up = l < L - 1;
  if (has_lo) stage_vec<R, CG>(v_lo, src + (l - 1) * m, m, lane);
  if (has_up) stage_vec<R, CG>(v_up, src_up + (l + 1) * m, m, lane);
  __syncwarp();
  double acc[R];
  zero_acc<R>(acc);
  if (has_lo) gemv_acc<R>(acc, A + (size_t)l * ms, v_lo, 0, m, m, lane);
  if (has_up) gemv_acc<R>(acc, B + (size_t)l * ms, v_up, 0, m, m, lane);
  if (far) far_terms<R, CG>(acc, far, xfar_lo, xfar_up, l, L, m, ms, v_lo, lane);
  if (!COUPLED) {
#pragma unroll
    for (int r = 0; r < R; ++r) v_g[lane + 32 * r] = acc[r];
    __syncwarp();
    zero_acc<R>(acc);
    gemv_acc<R>(acc, C + (size_t)l * ms, v_g, 0, m, m, lane);
  }
  double ls = 0.0;
  if (want_sum) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int row = lane + 32 * r;
      if (row < m) {
        dst[l * m + row] = acc[r];
        ls += acc[r];
      }
    }
    if (WARP_TOTAL) ls = warp_sum(ls);
  } else {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int row = lane + 32 * r;
      if (row < m) dst[l * m + row] = acc[r];
    }
  }
  __syncwarp();   // the slice is rewritten for the next level
  return ls;
}

// One level of the direct residual r_l = (Q^T x)_l = T_lo x_{l-1} + T_dd x_l +
// T_up x_{l+1} (Eq. (1)); returns ||r_l||_1 on every lane.  With q != NULL
// also stores q_l = (-T_dd)^{-1} r_l in FP32.
template <int R>
__device__ __forceinline__ double level_resid(const double* TLO, const double* TDD,
                                              const double* TUP, const double* NINV,
                                              const double* x, float* q, int64_t l, int64_t L,
                                              int m, int ms, double* slice, int lane,
                                              const FarDesc* far = nullptr) {
  constexpr int W = 32 * R;
  double* v_lo = slice;
  double* v_dd = slice + W;
  double* v_up = slice + 2 * W;
  if (l > 0) stage_vec<R>(v_lo, x + (l - 1) * m, m, lane);
  stage_vec<R>(v_dd, x + l * m, m, lane);
  if (l < L - 1) stage_vec<R>(v_up, x + (l + 1) * m, m, lane);
  __syncwarp();
  double acc[R];
  zero_acc<R>(acc);
  if (l > 0) {
    gemv_acc<R>(acc, TLO + (size_t)l * ms, v_lo, 0, m, m, lane);
  }
  gemv_acc<R>(acc, TDD + (size_t)l * ms, v_dd, 0, m, m, lane);
  if (l < L - 1) {
    gemv_acc<R>(acc, TUP + (size_t)l * ms, v_up, 0, m, m, lane);
  }
  if (far) far_terms<R>(acc, far, x, x, l, L, m, ms, v_lo, lane);
  double ls = 0.0;
#pragma unroll
  for (int r = 0; r < R; ++r) ls += fabs(acc[r]);
  const double total = warp_sum(ls);
  if (q) {
    __syncwarp();
#pragma unroll
    for (int r = 0; r < R; ++r) v_lo[lane + 32 * r] = acc[r];
    __syncwarp();
    zero_acc<R>(acc);
    gemv_acc<R>(acc, NINV + (size_t)l * ms, v_lo, 0, m, m, lane);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int row = lane + 32 * r;
      if (row < m) q[l * m + row] = (float)acc[r];
    }
  }
  __syncwarp();
  return total;
}

}  // namespace dev
}  // namespace mc
