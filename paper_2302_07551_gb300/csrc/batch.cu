// Batched kernels of the solve server (see batch.cuh): the per-level bodies
// of the single-chain kernels (level_sweep2, level_resid, level_sweep_lp)
// applied to every level of every active request in one persistent launch.
#include <cuda_bf16.h>
#include <math.h>

#include <type_traits>

#include "batch.cuh"
#include "lowprec_dev.cuh"
#include "lpteam_dev.cuh"
#include "resident_dev.cuh"
#include "sweep_dev.cuh"
#include "team_dev.cuh"
#include "wave_dev.cuh"

namespace mc {

namespace {

using namespace dev;

// Largest r in [lo, hi) with off[r] <= i (off is non-decreasing).
__device__ __forceinline__ int find_req(const int64_t* off, int lo, int hi, int64_t i) {
  hi -= 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (off[mid] <= i)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

// Request range [r0, r1) of the size classes [c0, c1) (the table is ordered
// by class).
__device__ __forceinline__ void class_range(const BTable* t, int c0, int c1, int& r0, int& r1) {
  r0 = c0 == 0 ? 0 : t->cls_end[c0 - 1];
  r1 = t->cls_end[c1 - 1];
}

constexpr unsigned long long kWaitNs = 2000000000ull;   // bound of one neighbour wait

// Unit q of a fused chunk of K sweeps over one bucket: sweep k, half-sweep h,
// request r and its levels l, l + 2, ..., l + 2 (n - 1) (a group of at most
// the request's G levels of one half-sweep: half-sweep 1 groups [a0, a1) of
// off_h1, then half-sweep 2 groups [b0, b1) of off_h2).
struct BUnit {
  int64_t k, l;
  int r, n;
  bool h2;
};

__device__ __forceinline__ BUnit unit_of(const BTable* t, unsigned long long q, int64_t n1,
                                         int64_t U, int64_t a0, int64_t b0, int r0, int r1) {
  BUnit u;
  u.k = (int64_t)(q / (unsigned long long)U);
  const int64_t rr = (int64_t)q - u.k * U;
  u.h2 = rr >= n1;
  const int64_t* off = u.h2 ? t->off_h2 : t->off_h1;
  const int64_t i = u.h2 ? b0 + (rr - n1) : a0 + rr;
  u.r = find_req(off, r0, r1, i);
  const BReq* Q = &t->r[u.r];
  const int par = u.h2 ? 1 - Q->p1 : Q->p1;
  const int64_t P = (Q->L - par + 1) / 2;        // levels of this half-sweep
  const int64_t g = i - off[u.r];
  const int G = Q->G;
  u.l = 2 * G * g + par;
  const int64_t left = P - (int64_t)G * g;
  u.n = left < G ? (int)left : G;
  return u;
}

// One level (m <= 32, lane = row) with every sum in the order of the resident kernels:
// S column groups, column j in group j % S, the terms of A and B in turn; the groups'
// sums added by a tree (rows shared by lanes) or in order (by warps); the level's sum
// row by row.
template <int S, bool TREE, bool COUPLED>
__device__ __forceinline__ double level_grouped(const BReq* Q, const double* src, double* dst,
                                                int64_t l, double* slice, int lane,
                                                bool want_sum) {
  static_assert(S == 1 || S == 2 || S == 4, "");
  constexpr int U = 8;
  const int m = Q->m;
  const bool has_lo = l > 0, has_up = l < Q->L - 1, in = lane < m;
  double *lo = slice, *up = slice + 32, *g = slice + 64;
  lo[lane] = has_lo && in ? __ldcg(src + (l - 1) * m + lane) : 0.0;
  up[lane] = has_up && in ? __ldcg(src + (l + 1) * m + lane) : 0.0;
  __syncwarp();
  auto total = [](const double (&p)[S]) {
    if constexpr (S == 1)
      return p[0];
    else if constexpr (S == 2)
      return p[0] + p[1];
    else if constexpr (TREE)
      return (p[0] + p[1]) + (p[2] + p[3]);
    else
      return ((p[0] + p[1]) + p[2]) + p[3];
  };
  double p[S];
#pragma unroll
  for (int s = 0; s < S; ++s) p[s] = 0.0;
  const double* A = Q->A + (size_t)l * Q->ms + lane;
  const double* B = Q->B + (size_t)l * Q->ms + lane;
  for (int j0 = 0; j0 < m; j0 += U) {
    double a[U], b[U];
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const bool ok = in && j0 + q < m;
      a[q] = ok && has_lo ? ld_stream(A + (size_t)(j0 + q) * m) : 0.0;
      b[q] = ok && has_up ? ld_stream(B + (size_t)(j0 + q) * m) : 0.0;
    }
#pragma unroll
    for (int q = 0; q < U; ++q) {
      p[q % S] = fma(a[q], lo[j0 + q], p[q % S]);
      p[q % S] = fma(b[q], up[j0 + q], p[q % S]);
    }
  }
  double v = total(p);
  if constexpr (!COUPLED) {
    g[lane] = v;
    __syncwarp();
#pragma unroll
    for (int s = 0; s < S; ++s) p[s] = 0.0;
    const double* C = Q->C + (size_t)l * Q->ms + lane;
    for (int j0 = 0; j0 < m; j0 += 2 * U) {
      double c[2 * U];
#pragma unroll
      for (int q = 0; q < 2 * U; ++q)
        c[q] = in && j0 + q < m ? ld_stream(C + (size_t)(j0 + q) * m) : 0.0;
#pragma unroll
      for (int q = 0; q < 2 * U; ++q) p[q % S] = fma(c[q], g[j0 + q], p[q % S]);
    }
    v = total(p);
  }
  if (in) dst[l * m + lane] = v;
  double sum = 0.0;
  if (want_sum) {
    __syncwarp();   // lo has been read
    lo[lane] = v;
    __syncwarp();
    if (lane == 0)
      for (int j = 0; j < m; ++j) sum += lo[j];
  }
  __syncwarp();   // the slice is rewritten for the next level
  return sum;
}

// Column groups of level l of a request in the resident order.
__device__ __forceinline__ int level_groups(const BReq* Q, int64_t l) {
  if (Q->res_s) return Q->res_s;
  const int C = Q->res_c, L = (int)Q->L, base = L / C, rem = L % C, long_end = (base + 1) * rem;
  const int r = l < long_end ? (int)l / (base + 1) : rem + ((int)l - long_end) / base;
  const int l0 = res::range_begin(L, C, r), n = res::range_begin(L, C, r + 1) - l0;
  const int t0 = (l0 ^ (int)l) & 1;   // the CTA's first level of this half-sweep
  return res::flat_split((n - t0 + 1) / 2 * Q->m);
}

template <bool COUPLED>
__device__ __forceinline__ double level_resident(const BReq* Q, const double* src, double* dst,
                                                 int64_t l, double* slice, int lane,
                                                 bool want_sum) {
  switch (level_groups(Q, l)) {
    case 1: return level_grouped<1, false, COUPLED>(Q, src, dst, l, slice, lane, want_sum);
    case 2: return level_grouped<2, false, COUPLED>(Q, src, dst, l, slice, lane, want_sum);
    default:
      return Q->res_s ? level_grouped<4, true, COUPLED>(Q, src, dst, l, slice, lane, want_sum)
                      : level_grouped<4, false, COUPLED>(Q, src, dst, l, slice, lane, want_sum);
  }
}

// K FP64 sweeps of the queue-path requests (b_path: m <= 16; build_table: m <= 32) in one launch.  Per
// request: sweep 0 reads x, sweeps 0..K-2 write xb in place, sweep K-1 writes z (so
// xb keeps the previous sweep for the step error).
template <bool COUPLED>
__global__ void __launch_bounds__(256, 4) k_b_sweeps(const BTable* __restrict__ t, int K,
                                                  unsigned long long* claim, BOut* out) {
  extern __shared__ double vsh[];
  const int lane = threadIdx.x & 31;
  double* slice = vsh + (threadIdx.x >> 5) * 3 * 32;
  int r0, r1;
  class_range(t, 0, 1, r0, r1);
  const int64_t a0 = t->off_h1[r0], a1 = t->off_h1[r1];
  const int64_t b0 = t->off_h2[r0], b1 = t->off_h2[r1];
  const int64_t n1 = a1 - a0, U = n1 + (b1 - b0);
  if (U == 0) return;
  const unsigned long long total = (unsigned long long)K * (unsigned long long)U;
  const int base = t->epoch;
  unsigned long long q0 = claim_unit(claim, lane);
  unsigned long long q = __shfl_sync(kFull, q0, 0);
  while (q < total) {
    q0 = claim_unit(claim, lane);
    const BUnit u = unit_of(t, q, n1, U, a0, b0, r0, r1);
    const BReq* Q = &t->r[u.r];
    const bool last = u.k == K - 1;
    double* dst = last ? Q->z : Q->xb;
    const double* src = u.h2 ? dst : (u.k == 0 ? Q->x : Q->xb);
    if (u.h2 || u.k > 0)
      wait_levels(Q->ver, u.l - 1, 2, u.n + 1, Q->L, base + (int)(u.h2 ? u.k + 1 : u.k),
                  &out[u.r].status, lane, kWaitNs);
    const bool want = u.k >= K - 2;   // e^T z of the last two sweeps only
    for (int i = 0; i < u.n; ++i) {
      const int64_t l = u.l + 2 * i;
      const double ls =
          Q->res_c ? level_resident<COUPLED>(Q, src, dst, l, slice, lane, want)
                   : level_sweep2<1, COUPLED, true, true>(Q->A, Q->B, Q->C, src, src, dst, l, Q->L,
                                                          Q->m, Q->ms, slice, lane, nullptr, nullptr,
                                                          nullptr, want);
      if (want && lane == 0) Q->lsum2[(u.k & 1) * Q->L + l] = ls;
    }
    publish_levels(Q->ver, u.l, 2, u.n, base + (int)u.k + 1, lane);
    q = __shfl_sync(kFull, q0, 0);
  }
}

// Direct residual of every request of the size classes up to m <= 128
// (LARGE = false) or m > 128 (LARGE = true).
template <bool LARGE>
__global__ void __launch_bounds__(256) k_b_resid(const BTable* __restrict__ t, int with_q) {
  extern __shared__ double vsh[];
  constexpr int RMAX = LARGE ? 8 : 4;
  const int lane = threadIdx.x & 31;
  double* slice = vsh + (threadIdx.x >> 5) * 3 * 32 * RMAX;
  const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  int r0, r1;
  class_range(t, LARGE ? 3 : 0, LARGE ? 4 : 3, r0, r1);
  const int64_t i0 = t->off_lv[r0], i1 = t->off_lv[r1];
  for (int64_t i = i0 + gw; i < i1; i += nw) {
    const int r = find_req(t->off_lv, r0, r1, i);
    const BReq* q = &t->r[r];
    const int64_t l = i - t->off_lv[r];
    float* qv = with_q ? q->q : nullptr;
    double ls;
    if (LARGE) {
      ls = level_resid<8>(q->TLO, q->TDD, q->TUP, q->NINV, q->x, qv, l, q->L, q->m, q->ms, slice, lane);
    } else {
      switch ((q->m + 31) / 32) {
        case 1: ls = level_resid<1>(q->TLO, q->TDD, q->TUP, q->NINV, q->x, qv, l, q->L, q->m, q->ms, slice, lane); break;
        case 2: ls = level_resid<2>(q->TLO, q->TDD, q->TUP, q->NINV, q->x, qv, l, q->L, q->m, q->ms, slice, lane); break;
        case 3: ls = level_resid<3>(q->TLO, q->TDD, q->TUP, q->NINV, q->x, qv, l, q->L, q->m, q->ms, slice, lane); break;
        default: ls = level_resid<4>(q->TLO, q->TDD, q->TUP, q->NINV, q->x, qv, l, q->L, q->m, q->ms, slice, lane); break;
      }
    }
    if (lane == 0) q->lsum[l] = ls;
  }
}

// which: 0 -> s = e^T z (with the breakdown check), 1 -> step, 2 -> residual,
// 3 -> e^T z of the last two sweeps of a fused chunk of K sweeps (from lsum2).
// One block per request (grid-stride), fixed order: thread k adds levels
// k, k + blockDim, ..., then a fixed shuffle tree.
__global__ void __launch_bounds__(256) k_b_reqsum(const BTable* __restrict__ t, BOut* out,
                                                  int which, int K = 1) {
  __shared__ double sh[32];
  for (int r = blockIdx.x; r < t->n; r += gridDim.x) {
    const BReq* q = &t->r[r];
    if (which == 3) {
      const double* a = q->lsum2 + ((K - 1) & 1) * q->L;
      const double* b = q->lsum2 + ((K - 2) & 1) * q->L;
      double va = 0.0, vb = 0.0;
      for (int64_t l = threadIdx.x; l < q->L; l += blockDim.x) {
        va += a[l];
        if (K >= 2) vb += b[l];
      }
      va = block_sum(va, sh);
      vb = block_sum(vb, sh);
      if (threadIdx.x == 0) {
        const double sp = K >= 2 ? vb : 1.0;
        out[r].s_last = va;
        out[r].s_prev = sp;
        out[r].s = va / sp;
        if (!(va > 0.0) || !isfinite(va) || !(sp > 0.0) || !isfinite(sp))
          out[r].status = MC_ERR_BREAKDOWN;
      }
      __syncthreads();
      continue;
    }
    double v = 0.0;
    for (int64_t l = threadIdx.x; l < q->L; l += blockDim.x) v += q->lsum[l];
    v = block_sum(v, sh);
    if (threadIdx.x == 0) {
      if (which == 0) {
        out[r].s = v;
        if (!(v > 0.0) || !isfinite(v)) out[r].status = MC_ERR_BREAKDOWN;
      } else if (which == 1) {
        out[r].step = v;
      } else {
        out[r].resid = v;
      }
    }
    __syncthreads();
  }
}

// x_l = src_l / s per level with the level's step error into lsum:
//   mode 0: src = z, s = e^T z, step against x;
//   mode 1: src = xb (refinement update), as mode 0;
//   mode 2: fused chunk of K sweeps: src = z / s_last, step against
//           x_prev / s_prev with x_prev = xb (K >= 2) or x (K = 1).
__global__ void __launch_bounds__(256) k_b_norm(const BTable* __restrict__ t, const BOut* out,
                                                int mode, int K = 1) {
  const int lane = threadIdx.x & 31;
  const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t tot = t->off_lv[t->n];
  for (int64_t i = gw; i < tot; i += nw) {
    const int r = find_req(t->off_lv, 0, t->n, i);
    const BReq* q = &t->r[r];
    const int64_t l = i - t->off_lv[r];
    const double inv = 1.0 / (mode == 2 ? out[r].s_last : out[r].s);
    const double pinv = mode == 2 ? 1.0 / out[r].s_prev : 1.0;
    const double* src = mode == 1 ? q->xb : q->z;
    const double* prev = (mode == 2 && K >= 2) ? q->xb : q->x;
    double e = 0.0;
    for (int k = lane; k < q->m; k += 32) {
      const int64_t j = l * q->m + k;
      const double p = src[j] * inv;
      e += fabs(p - prev[j] * pinv);
      q->x[j] = p;
    }
    e = warp_sum(e);
    if (lane == 0) q->lsum[l] = e;
  }
}

// Refinement update per level: xb = x + d, level sum into lsum.
__global__ void __launch_bounds__(256) k_b_update(const BTable* __restrict__ t) {
  const int lane = threadIdx.x & 31;
  const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t tot = t->off_lv[t->n];
  for (int64_t i = gw; i < tot; i += nw) {
    const int r = find_req(t->off_lv, 0, t->n, i);
    const BReq* q = &t->r[r];
    const int64_t l = i - t->off_lv[r];
    double e = 0.0;
    for (int k = lane; k < q->m; k += 32) {
      const int64_t j = l * q->m + k;
      const double v = q->x[j] + (double)q->d[j];
      q->xb[j] = v;
      e += v;
    }
    e = warp_sum(e);
    if (lane == 0) q->lsum[l] = e;
  }
}

__global__ void __launch_bounds__(256) k_b_zero_d(const BTable* __restrict__ t) {
  const int lane = threadIdx.x & 31;
  const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t tot = t->off_lv[t->n];
  for (int64_t i = gw; i < tot; i += nw) {
    const int r = find_req(t->off_lv, 0, t->n, i);
    const BReq* q = &t->r[r];
    if (q->path != kPathQueue) continue;
    const int64_t l = i - t->off_lv[r];
    for (int k = lane; k < q->m; k += 32) q->d[l * q->m + k] = 0.0f;
  }
}

// Low-precision correction sweeps of one bucket (size classes [c0, c1)), all
// K sweeps of a refinement step in one launch, d in place.  Paths by the
// request's block size: m <= 64 -> 16-byte lane loads, BW loads in flight,
// several lanes per column; 64 < m <= 128 -> G = GF = 2 (FP32 or two-row
// BF16); m > 128 -> FP32 G = 4, four-row BF16 G = 2, GF = 4.  CLS bounds the
// paths a kernel holds (0: m <= 64, 1: m <= 128, 2: m > 128), so that each
// kernel has the register count of its largest path.
template <typename TS, typename TL, bool COUPLED, int CLS, int BW>
__global__ void __launch_bounds__(256) k_b_sweeps_lp(const BTable* __restrict__ t, int K, int c0,
                                                     int c1, unsigned long long* claim,
                                                     BOut* out) {
  extern __shared__ float fsh[];
  constexpr int SL = CLS == 2 ? 256 : 128;
  const int lane = threadIdx.x & 31;
  float* slice = fsh + (threadIdx.x >> 5) * 3 * SL;
  int r0, r1;
  class_range(t, c0, c1, r0, r1);
  const int64_t a0 = t->off_h1[r0], a1 = t->off_h1[r1];
  const int64_t b0 = t->off_h2[r0], b1 = t->off_h2[r1];
  const int64_t n1 = a1 - a0, U = n1 + (b1 - b0);
  if (U == 0) return;
  const unsigned long long total = (unsigned long long)K * (unsigned long long)U;
  const int base = t->epoch;
  unsigned long long q0 = claim_unit(claim, lane);
  unsigned long long q = __shfl_sync(kFull, q0, 0);
  while (q < total) {
    q0 = claim_unit(claim, lane);
    const BUnit u = unit_of(t, q, n1, U, a0, b0, r0, r1);
    const BReq* Q = &t->r[u.r];
    if (u.h2 || u.k > 0)
      wait_levels(Q->ver, u.l - 1, 2, u.n + 1, Q->L, base + (int)(u.h2 ? u.k + 1 : u.k),
                  &out[u.r].status, lane, kWaitNs);
    for (int i = 0; i < u.n; ++i) {
      const int64_t l = u.l + 2 * i;
      // the path follows the request's m alone (never the bucket), so every
      // bucketing computes a level with the same arithmetic
      if constexpr (CLS == 2) {
        constexpr int GL = Pack<TL>::V == 2 ? 4 : 2;
        level_sweep_lp<TL, GL, 4, COUPLED, true>((const TL*)Q->lA, (const TL*)Q->lB, Q->lC,
                                                 Q->sc, Q->d, Q->q, l, Q->L, Q->m, Q->lp_bs,
                                                 Q->lp_cbs, slice, lane);
      } else if (CLS == 1 && Q->m > 64) {
        level_sweep_lp<TS, 2, 2, COUPLED, true>((const TS*)Q->lA, (const TS*)Q->lB, Q->lC,
                                                Q->sc, Q->d, Q->q, l, Q->L, Q->m, Q->lp_bs,
                                                Q->lp_cbs, slice, lane);
      } else if (sizeof(TS) == 4 || Q->m % 8 == 0) {
        // 16-byte lane loads (BF16 columns 16-byte aligned when m % 8 == 0)
        using S = typename std::conditional<sizeof(TS) == 4 && !std::is_same<TS, Bf16x2>::value,
                                            float, unsigned short>::type;
        if (Q->m <= 16)
          level_sweep_lp_small<S, 16, COUPLED, true, BW>((const S*)Q->lA, (const S*)Q->lB,
                                                         Q->lC, Q->sc, Q->d, Q->q, l, Q->L, Q->m,
                                                         Q->lp_bs, Q->lp_cbs, slice, lane);
        else if (Q->m <= 32)
          level_sweep_lp_small<S, 32, COUPLED, true, BW>((const S*)Q->lA, (const S*)Q->lB,
                                                         Q->lC, Q->sc, Q->d, Q->q, l, Q->L, Q->m,
                                                         Q->lp_bs, Q->lp_cbs, slice, lane);
        else
          level_sweep_lp_small<S, 64, COUPLED, true, BW>((const S*)Q->lA, (const S*)Q->lB,
                                                         Q->lC, Q->sc, Q->d, Q->q, l, Q->L, Q->m,
                                                         Q->lp_bs, Q->lp_cbs, slice, lane);
      } else {
        level_sweep_lp<TS, 1, 1, COUPLED, true>((const TS*)Q->lA, (const TS*)Q->lB, Q->lC,
                                                Q->sc, Q->d, Q->q, l, Q->L, Q->m, Q->lp_bs,
                                                Q->lp_cbs, slice, lane);
      }
    }
    publish_levels(Q->ver, u.l, 2, u.n, base + (int)u.k + 1, lane);
    q = __shfl_sync(kFull, q0, 0);
  }
}

// Correction sweeps of the team-path requests of one size class: units are single
// levels in the order (sweep, half-sweep, request, level), claimed by teams of TW
// warps.  Versions go on from chunk to chunk (the epoch), so the words need no
// reset.
template <typename S, int ROWS, int TW, bool COUPLED>
__global__ void __launch_bounds__(256, 2) k_b_team(const BTable* __restrict__ t, int K, int cls,
                                                   unsigned long long* claim, BOut* out) {
  extern __shared__ __align__(16) unsigned char lp_smem[];
  if ((int)blockIdx.x >= t->team_ctas[cls]) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int team = warp / TW, w = warp % TW, tt = threadIdx.x - team * TW * 32, bar = 1 + team;
  auto& sh = reinterpret_cast<LpTeamShared<ROWS, TW>*>(lp_smem)[team];
  int r0, r1;
  class_range(t, cls, cls + 1, r0, r1);
  const int64_t a0 = t->off_t1[r0], b0 = t->off_t2[r0];
  const int64_t n1 = t->off_t1[r1] - a0, U = n1 + (t->off_t2[r1] - b0);
  const unsigned long long total = (unsigned long long)K * (unsigned long long)U;
  const int base = t->epoch;
  unsigned long long q0 = w == 0 ? claim_unit(claim, lane) : 0ull, q;
  if (w == 0 && lane == 0) sh.next[1] = q0;
  if (w == 0) q0 = claim_unit(claim, lane);
  team_sync<TW>(bar);
  q = sh.next[1];
  int turn = 0;
  while (q < total) {
    unsigned long long qn = 0ull;
    if (w == 0 && lane == 0) sh.next[turn] = q0;
    const int64_t k = (int64_t)(q / (unsigned long long)U), rr = (int64_t)q - k * U;
    const bool h2 = rr >= n1;
    const int64_t* off = h2 ? t->off_t2 : t->off_t1;
    const int64_t i = h2 ? b0 + (rr - n1) : a0 + rr;
    const int r = find_req(off, r0, r1, i);
    const BReq* Q = &t->r[r];
    const LpLevels v{Q->lA, Q->lB, Q->lC, Q->sc, Q->q, Q->dv, Q->d, Q->L, Q->lp_bs, Q->lp_cbs,
                     Q->m};
    const LpUnit u{2 * (i - off[r]) + (h2 ? 1 - Q->p1 : Q->p1), base + (int)(h2 ? k + 1 : k),
                   base + (int)k + 1, k == 0 && !h2, k == K - 1};
    LpAhead<S, ROWS, TW, COUPLED> p;
    p.load(v, u, w, tt, lane);
    lp_team_unit<S, ROWS, TW, COUPLED>(v, sh, u, p, w, tt, lane, bar, &out[r].status, kWaitNs,
                                       [&]() {
                                         qn = sh.next[turn];
                                         turn ^= 1;
                                         if (w == 0) q0 = claim_unit(claim, lane);
                                       });
    q = qn;
  }
}

// FP64 sweeps of the team-path requests of one size class, one row per lane (as
// k_sweeps).  Bound by the unit's latency where a batch has fewer levels than
// teams, by HBM and the FP64 pipe elsewhere.  Against one warp per unit of 4 to 16
// levels on the FP64 pipe alone, a chunk of 64 sweeps: 2000 x 32 + 1500 x 16 +
// 2500 x 24 coupled 3.20 -> 1.41 ms, 4000 x 64 inverse 8.43 -> 4.46, eight requests
// of 16 to 128 rows coupled 9.9 -> 4.5, four of 48 to 200 rows 37.8 -> 6.4.
template <int TW, bool COUPLED>
__global__ void __launch_bounds__(256, 3) k_b_team64(const BTable* __restrict__ t, int K, int cls,
                                                     unsigned long long* claim, BOut* out) {
  extern __shared__ __align__(16) unsigned char team_smem[];
  if ((int)blockIdx.x >= t->team_ctas[cls]) return;
  using Sh = TeamShared<TW, 1>;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int team = warp / TW, w = warp % TW, tt = threadIdx.x - team * TW * 32, bar = 1 + team;
  const int row0 = 32 * w;
  Sh& sh = reinterpret_cast<Sh*>(team_smem)[team];
  int r0, r1;
  class_range(t, cls, cls + 1, r0, r1);
  const int64_t a0 = t->off_t1[r0], b0 = t->off_t2[r0];
  const int64_t n1 = t->off_t1[r1] - a0, U = n1 + (t->off_t2[r1] - b0);
  const unsigned long long total = (unsigned long long)K * (unsigned long long)U;
  unsigned long long q0 = w == 0 ? claim_unit(claim, lane) : 0ull, q;
  if (w == 0 && lane == 0) sh.next[1] = q0;
  if (w == 0) q0 = claim_unit(claim, lane);
  team_sync<TW>(bar);
  q = sh.next[1];
  int turn = 0, s = 0;
  while (q < total) {
    if (w == 0 && lane == 0) sh.next[turn] = q0;
    const int64_t k = (int64_t)(q / (unsigned long long)U), rr = (int64_t)q - k * U;
    const bool h2 = rr >= n1;
    const int64_t* off = h2 ? t->off_t2 : t->off_t1;
    const int64_t i = h2 ? b0 + (rr - n1) : a0 + rr;
    const int r = find_req(off, r0, r1, i);
    const BReq* Q = &t->r[r];
    const int64_t l = 2 * (i - off[r]) + (h2 ? 1 - Q->p1 : Q->p1), L = Q->L;
    const int m = Q->m;
    const size_t at = (size_t)l * Q->ms;
    const bool has_lo = l > 0, has_up = l < L - 1;
    double* dst = k == K - 1 ? Q->z : Q->xb;
    const double* src = h2 ? dst : (k == 0 ? Q->x : Q->xb);
    const int2 ea = Q->eA[l], eb = Q->eB[l], ec = COUPLED ? make_int2(0, 0) : Q->eC[l];
    if (h2 || k > 0)
      wait_neighbours(Q->ver, l, L, (Q->vbase + (int)(h2 ? k + 1 : k)) * TW, &out[r].status, lane,
                      kWaitNs);
    const double x0[1] = {has_lo && tt < m ? __ldcg(src + (l - 1) * m + tt) : 0.0};
    const double x1[1] = {has_up && tt < m ? __ldcg(src + (l + 1) * m + tt) : 0.0};
    stage_rows<1>(sh.slot[s].v[0], sh.slot[s].x[0], sh.exps[s][0], x0, m, tt, 32, w, lane);
    stage_rows<1>(sh.slot[s].v[1], sh.slot[s].x[1], sh.exps[s][1], x1, m, tt, 32, w, lane);
    team_sync<TW>(bar);
    const unsigned long long qn = sh.next[turn];
    turn ^= 1;
    if (w == 0) q0 = claim_unit(claim, lane);
    double acc[1] = {0.0};
    if (has_lo)
      rows_product<1, 0>(acc, Q->A + at, sh.slot[s].v[0], sh.slot[s].x[0], ea,
                         team_exp<TW>(sh.exps[s][0]), 0, m, m, row0, lane);
    if (has_up)
      rows_product<1, 0>(acc, Q->B + at, sh.slot[s].v[1], sh.slot[s].x[1], eb,
                         team_exp<TW>(sh.exps[s][1]), 0, m, m, row0, lane);
    if constexpr (!COUPLED) {
      s ^= 1;
      stage_rows<1>(sh.slot[s].v[0], sh.slot[s].x[0], sh.exps[s][0], acc, m, row0 + lane, 32, w,
                    lane);
      team_sync<TW>(bar);
      acc[0] = 0.0;
      rows_product<1, 0>(acc, Q->C + at, sh.slot[s].v[0], sh.slot[s].x[0], ec,
                         team_exp<TW>(sh.exps[s][0]), 0, m, m, row0, lane);
    }
    double ls = 0.0;
    if (row0 + lane < m) {
      dst[l * m + row0 + lane] = acc[0];
      ls = acc[0];
    }
    __threadfence();
    __syncwarp();
    if (lane == 0) red_release(Q->ver + l, 1);
    if (k >= K - 2) {   // e^T z of the last two sweeps only
      ls = team_total<TW>(warp_sum(ls), sh.part, w, lane, bar);
      if (w == 0 && lane == 0) Q->lsum2[(k & 1) * L + l] = ls;
    }
    s ^= 1;
    q = qn;
  }
}

template <bool C>
cudaError_t team64_launches(const BTable* t, unsigned long long* claim, BOut* out, int paths,
                            int K, int sms, cudaStream_t b0, const cudaStream_t* b) {
  const int n = 3 * sms;
  if (paths & path_bit(kPathTeam, 0))
    k_b_team64<1, C><<<n, 256, 8 * sizeof(TeamShared<1, 1>), b0>>>(t, K, 0, claim, out);
  if (paths & path_bit(kPathTeam, 1))
    k_b_team64<2, C><<<n, 256, 4 * sizeof(TeamShared<2, 1>), b[0]>>>(t, K, 1, claim + 1, out);
  if (paths & path_bit(kPathTeam, 2))
    k_b_team64<4, C><<<n, 256, 2 * sizeof(TeamShared<4, 1>), b[1]>>>(t, K, 2, claim + 2, out);
  if (paths & path_bit(kPathTeam, 3))
    k_b_team64<8, C><<<n, 256, sizeof(TeamShared<8, 1>), b[2]>>>(t, K, 3, claim + 3, out);
  return cudaGetLastError();
}

template <typename S, bool C>
cudaError_t team_launches(const BTable* t, unsigned long long* claim, BOut* out, int paths, int K,
                          int sms, const cudaStream_t* b) {
  const int n = 2 * sms;
  if (paths & path_bit(kPathTeam, 1))
    k_b_team<S, 64, 4, C><<<n, 256, 2 * sizeof(LpTeamShared<64, 4>), b[0]>>>(t, K, 1, claim + 1,
                                                                            out);
  if (paths & path_bit(kPathTeam, 2))
    k_b_team<S, 128, 8, C><<<n, 256, sizeof(LpTeamShared<128, 8>), b[1]>>>(t, K, 2, claim + 2, out);
  if (paths & path_bit(kPathTeam, 3))
    k_b_team<S, 256, 8, C><<<n, 256, sizeof(LpTeamShared<256, 8>), b[2]>>>(t, K, 3, claim + 3, out);
  return cudaGetLastError();
}

template <typename K>
cudaError_t allow(K kernel, size_t bytes) {
  if (bytes <= 48 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <typename TS, typename TL, bool C>
cudaError_t lp_buckets(const BTable* t, unsigned long long* claim, BOut* out, int K, BTune g,
                       cudaStream_t s) {
  const BBuckets b = buckets_of(g.split64);
  const size_t sm_small = (size_t)(g.threads / 32) * 3 * 128 * sizeof(float);
  const size_t sm_large = (size_t)(g.threads / 32) * 3 * 256 * sizeof(float);
  cudaError_t e = allow(k_b_sweeps_lp<TS, TL, C, 2, 8>, sm_large);
  if (e != cudaSuccess) return e;
  for (int i = 0; i < b.n; ++i) {
    const int c0 = b.c0[i], c1 = b.c1[i];
    if (c1 <= 2) {          // m <= 64
      if (g.deep)
        k_b_sweeps_lp<TS, TL, C, 0, 16><<<g.blocks, g.threads, sm_small, s>>>(t, K, c0, c1,
                                                                            claim + i, out);
      else
        k_b_sweeps_lp<TS, TL, C, 0, 8><<<g.blocks, g.threads, sm_small, s>>>(t, K, c0, c1,
                                                                           claim + i, out);
    } else if (c1 <= 3) {   // m <= 128
      k_b_sweeps_lp<TS, TL, C, 1, 8><<<g.blocks, g.threads, sm_small, s>>>(t, K, c0, c1,
                                                                         claim + i, out);
    } else {
      k_b_sweeps_lp<TS, TL, C, 2, 8><<<g.blocks, g.threads, sm_large, s>>>(t, K, c0, c1,
                                                                         claim + i, out);
    }
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t b_sweeps(const BTable* t, unsigned long long* claim, BOut* out, int coupled, int K,
                     BTune g, cudaStream_t s) {
  const size_t sm = (size_t)(g.threads / 32) * 3 * 32 * sizeof(double);
  if (coupled)
    k_b_sweeps<true><<<g.blocks, g.threads, sm, s>>>(t, K, claim, out);
  else
    k_b_sweeps<false><<<g.blocks, g.threads, sm, s>>>(t, K, claim, out);
  return cudaGetLastError();
}

cudaError_t b_sweeps_finish(const BTable* t, BOut* out, int K, BTune g, cudaStream_t s) {
  k_b_reqsum<<<g.blocks, 256, 0, s>>>(t, out, 3, K);
  k_b_norm<<<g.blocks, g.threads, 0, s>>>(t, out, 2, K);
  k_b_reqsum<<<g.blocks, 256, 0, s>>>(t, out, 1);
  return cudaGetLastError();
}

cudaError_t b_resid(const BTable* t, BOut* out, int with_q, BTune g, cudaStream_t s) {
  const size_t sm_small = (size_t)(g.threads / 32) * 3 * 32 * 4 * sizeof(double);
  const size_t sm_large = (size_t)(g.threads / 32) * 3 * 32 * 8 * sizeof(double);
  cudaError_t e = allow(k_b_resid<true>, sm_large);
  if (e != cudaSuccess) return e;
  k_b_resid<false><<<g.blocks, g.threads, sm_small, s>>>(t, with_q);
  k_b_resid<true><<<g.blocks, g.threads, sm_large, s>>>(t, with_q);
  k_b_reqsum<<<g.blocks, 256, 0, s>>>(t, out, 2);
  return cudaGetLastError();
}

cudaError_t b_lp_zero(const BTable* t, BTune g, cudaStream_t s) {
  k_b_zero_d<<<g.blocks, g.threads, 0, s>>>(t);
  return cudaGetLastError();
}

cudaError_t b_lp_sweeps(const BTable* t, unsigned long long* t_claim, BOut* out, int bf16,
                        int coupled, int inner, BTune g, cudaStream_t s) {
  cudaError_t e;
  if (bf16)
    e = coupled ? lp_buckets<Bf16x2, __nv_bfloat16, true>(t, t_claim, out, inner, g, s)
                : lp_buckets<Bf16x2, __nv_bfloat16, false>(t, t_claim, out, inner, g, s);
  else
    e = coupled ? lp_buckets<float, float, true>(t, t_claim, out, inner, g, s)
                : lp_buckets<float, float, false>(t, t_claim, out, inner, g, s);
  return e;
}

int b_path(const Layout& y, int coupled, int num_sms) {
  if (resident_batch_group(y, coupled) >= 0) return kPathResident;
  if (y.lp == 0) return kPathTeam;   // (m <= 16: or the queue, by the batch)
  if (y.m <= 32) return kPathQueue;
  if ((y.lp == 1 || y.m % 8 == 0) &&
      y.L / 2 * (y.m <= 64 ? 4 : 8) <= 16ll * num_sms)   // as launch_sweeps_lp
    return kPathTeam;
  return kPathQueue;
}

cudaError_t b_team(const BTable* t, unsigned long long* team_claim, BOut* out, int paths,
                   int coupled, int K, int num_sms, cudaStream_t b0,
                   const cudaStream_t* b) {
  return coupled ? team64_launches<true>(t, team_claim, out, paths, K, num_sms, b0, b)
                 : team64_launches<false>(t, team_claim, out, paths, K, num_sms, b0, b);
}

cudaError_t b_lp_team(const BTable* t, unsigned long long* team_claim, BOut* out, int paths,
                      int bf16, int coupled, int inner, int num_sms, const cudaStream_t* b) {
  if (bf16)
    return coupled ? team_launches<unsigned short, true>(t, team_claim, out, paths, inner, num_sms, b)
                   : team_launches<unsigned short, false>(t, team_claim, out, paths, inner, num_sms, b);
  return coupled ? team_launches<float, true>(t, team_claim, out, paths, inner, num_sms, b)
                 : team_launches<float, false>(t, team_claim, out, paths, inner, num_sms, b);
}

cudaError_t b_lp_finish(const BTable* t, BOut* out, BTune g, cudaStream_t s) {
  k_b_update<<<g.blocks, g.threads, 0, s>>>(t);
  k_b_reqsum<<<g.blocks, 256, 0, s>>>(t, out, 0);
  k_b_norm<<<g.blocks, g.threads, 0, s>>>(t, out, 1);
  k_b_reqsum<<<g.blocks, 256, 0, s>>>(t, out, 1);
  return cudaGetLastError();
}

}  // namespace mc
