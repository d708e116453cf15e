// Low-precision correction sweeps of chains with fewer levels than the GPU has
// warps: what counts is the time of one unit (one level of one half-sweep),
// since a half-sweep's units all run at once and the next half-sweep waits for
// them.
//
//   * A team of TW warps owns the level; warp w takes a contiguous range of
//     the columns of every block, so a level of 262 KB (m = 256, BF16 coupled)
//     is streamed by 8 warps instead of one.  Partial sums of all rows are
//     added in warp order through shared memory.
//   * The operators do not depend on the neighbours: the first batch of every
//     operator's columns is in flight while the team waits for the words.
//   * The correction travels as 64-bit words {value, version} (version k + 1
//     after sweep k): the readers poll the words themselves, so that a version
//     costs one store and one load through L2 instead of a fence, a counter
//     release, a poll, an acquire and the load of the vector.  A word is
//     overwritten by the next version only after both neighbours have
//     published versions computed from it (the dataflow of fused.cu).
//
// 512 levels of 256, BF16 coupled: 71 -> 18.7 us a sweep (7.2 TB/s; 134 MB, more
// than L2 holds); 500 levels of 64, FP32 inverse: 17.8 -> 3.3; 500 of 128, BF16
// coupled: 32.6 -> 4.3.
//
// Lane loads are 16 bytes: E rows per lane, LPC lanes per column, CPW columns
// per warp load, RG row groups (FP32, m > 128).  BF16 needs m % 8 == 0.
#pragma once
#include "lowprec_dev.cuh"
#include "wave_dev.cuh"

namespace mc {
namespace dev {

template <typename S, int ROWS>
struct WideLane {
  static constexpr int E = 16 / (int)sizeof(S);
  static constexpr int LPC = ROWS / E < 32 ? ROWS / E : 32;
  static constexpr int RG = ROWS / (E * LPC);
  static constexpr int CPW = 32 / LPC;
};

// One batch of columns of one operator: at most 8 loads of 16 bytes in flight
// per lane, no more than the warp's CW columns need.
template <typename S, int ROWS, int CW>
struct WideBatch {
  static constexpr int RG = WideLane<S, ROWS>::RG, CPW = WideLane<S, ROWS>::CPW;
  static constexpr int WANT = CW / CPW > 0 ? CW / CPW : 1;
  static constexpr int NB = WANT < 8 / RG ? WANT : 8 / RG;
  static constexpr int COLS = NB * CPW;   // columns per batch (at most 64)
  uint4 t[NB][RG];
};

template <typename S, int ROWS, int CW>
__device__ __forceinline__ void wide_load(WideBatch<S, ROWS, CW>& w, const S* __restrict__ M,
                                          int j0, int j1, int m, int lane) {
  using P = WideLane<S, ROWS>;
  const int c = lane / P::LPC, r0 = P::E * (lane % P::LPC);
#pragma unroll
  for (int b = 0; b < WideBatch<S, ROWS, CW>::NB; ++b)
#pragma unroll
    for (int g = 0; g < P::RG; ++g) {
      const int j = j0 + b * P::CPW + c, row = r0 + g * P::E * P::LPC;
      w.t[b][g] = (j < j1 && row < m)
                      ? __ldcs(reinterpret_cast<const uint4*>(M + (size_t)j * m + row))
                      : make_uint4(0u, 0u, 0u, 0u);
    }
}

// acc += batch * v (v: shared, zero beyond m, readable to the batch's end).
template <typename S, int ROWS, int CW>
__device__ __forceinline__ void wide_fma(float (&acc)[WideLane<S, ROWS>::RG][WideLane<S, ROWS>::E],
                                         const WideBatch<S, ROWS, CW>& w, const float* v, int j0,
                                         int lane) {
  using P = WideLane<S, ROWS>;
  const int c = lane / P::LPC;
#pragma unroll
  for (int b = 0; b < WideBatch<S, ROWS, CW>::NB; ++b) {
    const float vj = v[j0 + b * P::CPW + c];
#pragma unroll
    for (int g = 0; g < P::RG; ++g)
#pragma unroll
      for (int e = 0; e < P::E; ++e)
        acc[g][e] = fmaf(small_elem(w.t[b][g], e, S()), vj, acc[g][e]);
  }
}

// Columns [j0, j1), at most CW of them, whose first batch is already in `w`.
template <typename S, int ROWS, int CW>
__device__ __forceinline__ void wide_product(
    float (&acc)[WideLane<S, ROWS>::RG][WideLane<S, ROWS>::E], WideBatch<S, ROWS, CW>& w,
    const S* __restrict__ M, const float* v, int j0, int j1, int m, int lane) {
  constexpr int COLS = WideBatch<S, ROWS, CW>::COLS;
  int j = j0;
  if constexpr (COLS < CW) {
    for (; j + COLS < j1; j += COLS) {
      WideBatch<S, ROWS, CW> n;
      wide_load<S, ROWS, CW>(n, M, j + COLS, j1, m, lane);
      wide_fma<S, ROWS, CW>(acc, w, v, j, lane);
      w = n;
    }
  }
  wide_fma<S, ROWS, CW>(acc, w, v, j, lane);
}

// Sum over the lanes that share a row (fixed shuffle tree), then the warp's
// row sums into part (lanes of the first column).
template <typename S, int ROWS>
__device__ __forceinline__ void wide_store(
    float (&acc)[WideLane<S, ROWS>::RG][WideLane<S, ROWS>::E], float* part, int lane) {
  using P = WideLane<S, ROWS>;
#pragma unroll
  for (int o = P::LPC; o < 32; o <<= 1)
#pragma unroll
    for (int g = 0; g < P::RG; ++g)
#pragma unroll
      for (int e = 0; e < P::E; ++e) acc[g][e] += __shfl_xor_sync(0xffffffffu, acc[g][e], o);
  if (lane < P::LPC) {
#pragma unroll
    for (int g = 0; g < P::RG; ++g)
#pragma unroll
      for (int e = 0; e < P::E; e += 4)
        *reinterpret_cast<float4*>(part + P::E * lane + g * P::E * P::LPC + e) =
            make_float4(acc[g][e], acc[g][e + 1], acc[g][e + 2], acc[g][e + 3]);
  }
}

// The words at p and q (either may be NULL: zero) once they carry `version`
// (bounded: after wait_ns, or once a timeout is latched, MC_ERR_TIMEOUT is
// latched and the last values are taken).
__device__ __forceinline__ float2 wait_words(const unsigned long long* p,
                                             const unsigned long long* q, int version,
                                             int* status, unsigned long long wait_ns) {
  const unsigned long long want = (unsigned long long)(unsigned)version << 32;
  unsigned long long a = p ? ld_word(p) : want, b = q ? ld_word(q) : want;
  unsigned long long t0 = 0;
  for (int it = 0; (int)(a >> 32) != version || (int)(b >> 32) != version; ++it) {
    if (p) a = ld_word(p);
    if (q) b = ld_word(q);
    if (it == 0) {
      t0 = global_ns();
    } else if ((it & 63) == 0) {
      if (*reinterpret_cast<volatile int*>(status) == (int)MC_ERR_TIMEOUT) break;
      if (global_ns() - t0 > wait_ns) {
        atomicCAS(status, 0, (int)MC_ERR_TIMEOUT);
        break;
      }
    }
  }
  return make_float2(__uint_as_float((unsigned)a), __uint_as_float((unsigned)b));
}

// Shared memory of one team.  Rows and columns run to ROWS; the batches read v
// up to 63 entries further.
template <int ROWS, int TW>
struct alignas(16) LpTeamShared {
  float v[2][ROWS + 64];
  float g[ROWS + 64];
  float part[TW][ROWS];
  unsigned long long next[2];
};

// Operators and vectors of a chain (or one request of a batch).
struct LpLevels {
  const void* A;
  const void* B;
  const float* C;
  const float* sc;
  const float* q;
  unsigned long long* dv;   // {value, version}
  float* d;                 // the last sweep's values
  int64_t L, abs_, cbs;
  int m;
};

// First column of warp w's range: multiples of 16 columns, so that the ranges of
// every lane layout start on a whole load; at most ROWS / TW (>= 16) columns.
template <int TW>
__device__ __forceinline__ int lp_col(int m, int w) {
  const int cw = ((m + TW - 1) / TW + 15) / 16 * 16, j = w * cw;
  return j < m ? j : m;
}

// A unit: level l of one half-sweep, reading versions `need` of levels l - 1 and
// l + 1 (zero: the first half-sweep, whose start vector is zero and not read)
// and writing version `out` (last: the values as well).
struct LpUnit {
  int64_t l;
  int need, out;
  bool zero, last;
};

// What a unit needs besides its neighbours' words, loaded ahead of time: the
// first batch of each operator, the block scales and the right-hand side.
template <typename S, int ROWS, int TW, bool COUPLED>
struct LpAhead {
  static constexpr int CW = ROWS / TW;
  static_assert(CW >= 16 && ROWS <= 32 * TW, "ranges of whole loads, one row per thread");
  WideBatch<S, ROWS, CW> a, b;
  WideBatch<float, ROWS, CW> c;
  float s_lo, s_up, q;

  __device__ __forceinline__ void load(const LpLevels& v, const LpUnit& u, int w, int tt,
                                       int lane) {
    const int m = v.m, j0 = lp_col<TW>(m, w), j1 = u.zero ? j0 : lp_col<TW>(m, w + 1);
    wide_load<S, ROWS, CW>(a, reinterpret_cast<const S*>(v.A) + u.l * v.abs_, j0,
                           u.l > 0 ? j1 : j0, m, lane);
    wide_load<S, ROWS, CW>(b, reinterpret_cast<const S*>(v.B) + u.l * v.abs_, j0,
                           u.l < v.L - 1 ? j1 : j0, m, lane);
    if (!COUPLED) wide_load<float, ROWS, CW>(c, v.C + u.l * v.cbs, j0, j1, m, lane);
    s_lo = v.sc[2 * u.l];
    s_up = v.sc[2 * u.l + 1];
    q = tt < m ? v.q[u.l * m + tt] : 0.0f;
  }
};

// One unit by a team.  hand(): called by every thread after the first barrier.
template <typename S, int ROWS, int TW, bool COUPLED, typename H>
__device__ __forceinline__ void lp_team_unit(const LpLevels& a, LpTeamShared<ROWS, TW>& sh,
                                             const LpUnit& u, LpAhead<S, ROWS, TW, COUPLED>& p,
                                             int w, int tt, int lane, int bar, int* status,
                                             unsigned long long wait_ns, H hand) {
  constexpr int CW = ROWS / TW;
  const int m = a.m;
  const int64_t l = u.l;
  const bool has_lo = l > 0, has_up = l < a.L - 1;
  const int j0 = lp_col<TW>(m, w), j1 = lp_col<TW>(m, w + 1);
  if (!u.zero) {
    for (int i = tt; i < ROWS + 64; i += 32 * TW) {
      float2 v = make_float2(0.0f, 0.0f);
      if (i < m)
        v = wait_words(has_lo ? a.dv + (l - 1) * m + i : nullptr,
                       has_up ? a.dv + (l + 1) * m + i : nullptr, u.need, status, wait_ns);
      sh.v[0][i] = v.x * p.s_lo;
      sh.v[1][i] = v.y * p.s_up;
    }
  }
  team_sync<TW>(bar);
  hand();
  const float q = p.q;
  if (!u.zero) {
    using P = WideLane<S, ROWS>;
    float acc[P::RG][P::E];
#pragma unroll
    for (int g = 0; g < P::RG; ++g)
#pragma unroll
      for (int e = 0; e < P::E; ++e) acc[g][e] = 0.0f;
    if (j0 < j1) {
      if (has_lo)
        wide_product<S, ROWS, CW>(acc, p.a, reinterpret_cast<const S*>(a.A) + l * a.abs_, sh.v[0],
                                  j0, j1, m, lane);
      if (has_up)
        wide_product<S, ROWS, CW>(acc, p.b, reinterpret_cast<const S*>(a.B) + l * a.abs_, sh.v[1],
                                  j0, j1, m, lane);
    }
    wide_store<S, ROWS>(acc, sh.part[w], lane);
  }
  team_sync<TW>(bar);
  auto total = [&](int row) {
    float t = sh.part[0][row];
#pragma unroll
    for (int i = 1; i < TW; ++i) t += sh.part[i][row];
    return t;
  };
  if constexpr (!COUPLED) {
    if (!u.zero) {
      for (int i = tt; i < ROWS + 64; i += 32 * TW) sh.g[i] = i < m ? total(i) : 0.0f;
      team_sync<TW>(bar);
      using P = WideLane<float, ROWS>;
      float acc[P::RG][P::E];
#pragma unroll
      for (int g = 0; g < P::RG; ++g)
#pragma unroll
        for (int e = 0; e < P::E; ++e) acc[g][e] = 0.0f;
      if (j0 < j1)
        wide_product<float, ROWS, CW>(acc, p.c, a.C + l * a.cbs, sh.g, j0, j1, m, lane);
      wide_store<float, ROWS>(acc, sh.part[w], lane);
      team_sync<TW>(bar);
    }
  }
  if (tt < m) {
    const float v = (u.zero ? 0.0f : total(tt)) + q;
    st_word(a.dv + l * m + tt, __float_as_uint(v), (unsigned)u.out);
    if (u.last) a.d[l * m + tt] = v;
  }
}

}  // namespace dev
}  // namespace mc
