// Level products of the fused FP64 sweeps by teams of warps.
//
// A team of TW warps owns one unit (one level of one half-sweep).  Warp w owns
// the rows 32 RW w .. 32 RW (w + 1) - 1, RW = 1 or 2 per lane, of every block, so
// each block column is one coalesced 256-byte load per 32 rows, every
// multiply-add lands in the lane's own accumulators and no partial sums cross
// the warps; the neighbour vectors are staged once per team in shared memory.
// Splitting the rows of large blocks keeps 16 loads per lane in flight with
// 80 registers at any m, and shortens a unit's time, which is what a chain
// with few levels waits for.
//
// The multiply-adds are shared between the FP64 pipe and the integer pipes
// (fixed_dev.cuh), which moves the bound from the FP64 pipe (98 % busy, 74 % of
// the HBM copy rate) to HBM.  64 sweeps with residual units: L = 32768, m = 64
// 41.8 -> 29.5 ms (4.98 -> 7.1 TB/s streamed); 32 coupled sweeps, L = 5001,
// m = 100, 7.32 -> 5.47 ms; 16 sweeps of 4096 paired
// levels of 256, 19.2 -> 12.7 ms (one warp per level with 8 rows a lane: 21.2);
// block Hessenberg, L = 4096, 64 sweeps, 11.9 -> 8.0 ms (with four of eight
// entries on the integer pipes 8.3, L = 32768 unchanged).
#pragma once
#include "fixed_dev.cuh"
#include "sweep_dev.cuh"
#include "wave_dev.cuh"

namespace mc {
namespace dev {

// Which entries of a batch of `total` per lane go to the fixed-point
// accumulators: n8 of every 8, spread evenly.  Three of eight where every lane
// owns rows: the FP64 pipe then needs 10 clocks an entry and SM where
// streaming it at the read rate of HBM takes 10.7.  Four of eight where some
// lanes of the last 32-row group own none (their FP64 slots are lost).
__host__ __device__ constexpr bool fixed_slot(int idx, int total, int n8) {
  const int n = (n8 * total + 4) / 8;
  return ((idx + 1) * n) / total != (idx * n) / total;
}

template <int RW>
struct TeamTune {
  static constexpr int U = RW == 1 ? 16 : 8;   // columns per batch
};

// Threads per block and blocks per SM of a team kernel: 24 warps an SM.
template <int TW>
struct TeamBlock {
  static constexpr int T = (TW == 3 || TW == 6) ? 192 : 256;
  static constexpr int B = 768 / T;
};

// Vectors staged for one product: FP64 and integer forms, zero beyond m.
template <int W>
struct TeamSlot {
  double v[2][W];
  uint64_t x[2][W];
};

// acc[r] += sum over columns [j0b, j1) of M(row0 + lane + 32 r, j) v_j.  MC:
// the block size when it fills the team's rows (no bounds checks), else 0.
// etot = largest exponent of the block + of the vector.
template <int RW, int MC>
__device__ __forceinline__ void rows_mix(double (&acc)[RW], const double* __restrict__ M,
                                         const double* v, const uint64_t* xv, int etot, int j0b,
                                         int j1, int m_, int row0, int lane) {
  constexpr int U = TeamTune<RW>::U, T = U * RW, N8 = MC ? 3 : 4;
  const int m = MC ? MC : m_;
  uint32_t fa[RW][4];
#pragma unroll
  for (int r = 0; r < RW; ++r) fa[r][0] = fa[r][1] = fa[r][2] = fa[r][3] = 0u;
  const double* p = M + (size_t)j0b * m + row0 + lane;
#pragma unroll 1
  for (int j0 = j0b; j0 < j1; j0 += U, p += (size_t)U * m) {
    double t[U][RW];
#pragma unroll
    for (int q = 0; q < U; ++q)
#pragma unroll
      for (int r = 0; r < RW; ++r)
        t[q][r] = (MC || (j0 + q < j1 && row0 + lane + 32 * r < m))
                      ? ld_stream(p + (size_t)q * m + 32 * r)
                      : 0.0;
#pragma unroll
    for (int q = 0; q < U; q += 2) {
      const double2 vv = *reinterpret_cast<const double2*>(v + j0 + q);
      const ulonglong2 xx = *reinterpret_cast<const ulonglong2*>(xv + j0 + q);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const double vj = h ? vv.y : vv.x;
        const uint64_t xj = h ? xx.y : xx.x;
        const uint32_t xl = (uint32_t)xj & 0xfffff800u, xh = (uint32_t)(xj >> 32);
        const int b = etot - (int)((uint32_t)xj & 0x7ffu);
#pragma unroll
        for (int r = 0; r < RW; ++r) {
          if (fixed_slot((q + h) * RW + r, T, N8))
            fixed_fma(fa[r], t[q + h][r], xl, xh, b);
          else
            acc[r] = fma(t[q + h][r], vj, acc[r]);
        }
      }
    }
  }
  // truncations of up to m terms: below 2^-57 of the row's whole sum (fixed_safe)
#pragma unroll
  for (int r = 0; r < RW; ++r) acc[r] += fixed_part(fa[r], etot);
}

// As rows_mix on the FP64 pipe alone.
template <int RW, int MC>
__device__ __forceinline__ void rows_f64(double (&acc)[RW], const double* __restrict__ M,
                                         const double* v, int j0b, int j1, int m_, int row0,
                                         int lane) {
  constexpr int U = TeamTune<RW>::U;
  const int m = MC ? MC : m_;
  const double* p = M + (size_t)j0b * m + row0 + lane;
#pragma unroll 1
  for (int j0 = j0b; j0 < j1; j0 += U, p += (size_t)U * m) {
    double t[U][RW];
#pragma unroll
    for (int q = 0; q < U; ++q)
#pragma unroll
      for (int r = 0; r < RW; ++r)
        t[q][r] = (MC || (j0 + q < j1 && row0 + lane + 32 * r < m))
                      ? ld_stream(p + (size_t)q * m + 32 * r)
                      : 0.0;
#pragma unroll
    for (int q = 0; q < U; q += 2) {
      const double2 vv = *reinterpret_cast<const double2*>(v + j0 + q);
#pragma unroll
      for (int r = 0; r < RW; ++r) {
        acc[r] = fma(t[q][r], vv.x, acc[r]);
        acc[r] = fma(t[q + 1][r], vv.y, acc[r]);
      }
    }
  }
}

// acc += M v on both pipes where the exponents of block and vector allow it, else
// and for m <= 16 on the FP64 pipe alone: joining the two sums costs more than the
// few columns save.
template <int RW, int MC>
__device__ __forceinline__ void rows_product(double (&acc)[RW], const double* M, const double* v,
                                             const uint64_t* xv, int2 eb, int ev, int j0, int j1,
                                             int m, int row0, int lane) {
  if (m > 16 && fixed_safe(eb, ev))
    rows_mix<RW, MC>(acc, M, v, xv, eb.x + (ev & 0xfff), j0, j1, m, row0, lane);
  else
    rows_f64<RW, MC>(acc, M, v, j0, j1, m, row0, lane);
}

// Exponents over the team's warps.
template <int TW>
__device__ __forceinline__ int team_exp(const int* e) {
  int v = e[0];
#pragma unroll
  for (int i = 1; i < TW; ++i) v = exp_join(v, e[i]);
  return v;
}

// Rows first, first + stride, ... of one vector of m rows into a staged slot.
template <int RW>
__device__ __forceinline__ void stage_rows(double* v, uint64_t* x, int* exps,
                                           const double (&y)[RW], int m, int first, int stride,
                                           int w, int lane) {
  unsigned most = 0u, low = 0u;
  bool zero = false;
#pragma unroll
  for (int i = 0; i < RW; ++i) {
    v[first + stride * i] = y[i];
    x[first + stride * i] = fixed_entry(y[i]);
    most = max(most, exp_field(y[i]));
    low = max(low, exp_low(y[i]));
    zero = zero || (first + stride * i < m && is_zero(y[i]));
  }
  most = __reduce_max_sync(kFull, most);
  low = __reduce_max_sync(kFull, low);
  zero = __any_sync(kFull, zero);
  if (lane == 0) exps[w] = exp_pack(most, low, zero);
}

// Sum of the warps' values in warp order (valid on the team's first warp).
template <int TW>
__device__ __forceinline__ double team_total(double t, double* part, int w, int lane, int bar) {
  if constexpr (TW == 1) return t;
  if (lane == 0) part[w] = t;
  team_sync<TW>(bar);
  double v = part[0];
#pragma unroll
  for (int i = 1; i < TW; ++i) v += part[i];
  return v;
}

// Shared memory of one team: a ring of two staged products (a warp that writes
// slot i + 1 has passed the barrier of slot i, so every warp of the team has
// finished reading slot i - 1), the exponents found by each warp, the
// units to come, and partial level sums.
// The staged vectors are read in 16-byte pairs, so every team's slots start on a
// 16-byte boundary.
template <int TW, int RW>
struct alignas(16) TeamShared {
  TeamSlot<32 * RW * TW> slot[2];
  int exps[2][2][TW];
  unsigned long long next[2];
  double part[TW];
};

}  // namespace dev
}  // namespace mc
