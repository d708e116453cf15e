// Set-up kernels: block layout of Q^T, batched LU of the diagonal blocks and
// the operators that apply Q_{l,l}^{-1} in Algorithm 2 (steps 2 and 3).
#include <cooperative_groups.h>
#include <math.h>

#include <type_traits>

#include "fixed_dev.cuh"
#include "mc_internal.cuh"

namespace mc {

namespace {

// Exponents of a lane's entries of a block, joined over the lanes of `mask` and into
// its block_exp (the rows' part comes later, k_weak_rows).
struct Exps {
  unsigned most = 0u, low = 0u;
  __device__ __forceinline__ void take(double v) {
    most = max(most, dev::exp_field(v));
    low = max(low, dev::exp_low(v));
  }
  __device__ __forceinline__ void join(int2* to, bool first, unsigned mask = 0xffffffffu) {
    most = __reduce_max_sync(mask, most);
    low = __reduce_max_sync(mask, low);
    if (first) {
      atomicMax(&to->x, (int)most);
      atomicMax(&to->y, (int)low);
    }
  }
};

// Copy of one block (or of a 2048-entry chunk of it) by a warp, zero where the
// block is missing and beyond m * m.
constexpr int kChunk = 2048;
__device__ __forceinline__ Exps copy_chunk(const double* src, double* dst, int e0, int mm, int ms,
                                           int lane) {
  Exps x;
  const int e1 = min(e0 + kChunk, ms);
  for (int e = e0 + lane; e < e1; e += 8 * 32) {
    double v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = src && e + 32 * q < mm ? __ldcs(src + e + 32 * q) : 0.0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      if (e + 32 * q < e1) dst[e + 32 * q] = v[q];
      x.take(v[q]);
    }
  }
  return x;
}

// Planes TLO, TUP, TDD from the generator blocks (Sect. 2 block partition of
// Q^T).  A row-major Q block is the column-major storage of its transpose, so
// T_{l,l-1} = (Q_{l-1,l})^T is up[l-1] copied verbatim, T_{l,l+1} =
// (Q_{l+1,l})^T is dn[l+1], T_{l,l} = loc[l].  Missing boundary blocks and
// the padding beyond m*m are zero.  The exponents of TLO and TUP come with the
// copy, without another pass.
__global__ void __launch_bounds__(256) k_layout(const double* dn, const double* loc,
                                                const double* up, double* tlo, double* tup,
                                                double* tdd, int2* elo, int2* eup, int64_t L, int m,
                                                int ms) {
  const int64_t mm = (int64_t)m * m;
  const int chunks = (ms + kChunk - 1) / kChunk, lane = threadIdx.x & 31;
  const int64_t total = 3 * L * chunks, nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < total; t += nw) {
    const int64_t b = t / chunks, l = b / 3;
    const int p = (int)(b - 3 * l), e0 = (int)(t - b * chunks) * kChunk;
    const double* src = p == 0   ? (l > 0 ? up + (l - 1) * mm : nullptr)
                        : p == 1 ? (l < L - 1 ? dn + (l + 1) * mm : nullptr)
                                 : loc + l * mm;
    double* dst = (p == 0 ? tlo : p == 1 ? tup : tdd) + (size_t)l * ms;
    Exps x = copy_chunk(src, dst, e0, (int)mm, ms, lane);
    if (p < 2) x.join((p == 0 ? elo : eup) + l, lane == 0);
  }
}

// ---- LU and inverse by Gauss-Jordan elimination ------------------------------
//
// Step k of an in-place Gauss-Jordan inversion without pivoting updates the
// whole matrix by a rank-1 product of column k over the pivot and row k.  Row k
// from the diagonal on is U's row k at that moment and the scaled column below
// it is L's column k, so the factors come on the way.  Per block m^3
// multiply-adds, what LU and two triangular solves take, but in m equal steps
// of a full m x m update in which no thread idles and no triangle is walked.
//
// The matrix stays in registers: thread (ti, tj) of a G x G grid owns the
// entries (ti + G a, tj + G b), a, b < R.  A step: the owners of row and column k
// have put them into shared memory; one warp forms 1 / pivot and the scaled
// column (a division is a dozen FP64 instructions, 16 clocks each); everybody
// does R^2 multiply-adds; the owners put row and column k + 1 there.  Row k, column k
// and the pivot take their new values from the same update, with the
// multipliers -1/pivot for row k and 1 for column k and the old entries zero.
// A diagonal entry is kept in two parts, its value at the start (or the inverse
// pivot) and the sum of its updates, added where it is used: m updates rounded
// at the size of the dominant diagonal would be most of the inverse's error
// (relative error over 8192 blocks of 64: LU and solves 4.3e-16, this 2.0e-16).
// Whether a pivot vanishes is decided by plain LU: a block one of whose pivots
// cancels to below 2^-45 of its diagonal entry, or is no number, is given up here
// and formed again by plain_block, with true divisions (a / -a is -1, a * (1 / -a)
// need not be) and the diagonal in one part, so that two phases whose rates balance
// still meet their zero pivot and nothing else is refused.  8192 blocks of 64 take
// the same time with the check.
// Bound: the FP64 pipe (a tenth of its instructions are the pivot's).  8192 blocks
// of 64: 7.7 -> 4.65 ms (3.4 at the pipe's rate).
__device__ __forceinline__ bool cancels(double piv, double diag) {
  return (((unsigned)__double2hiint(piv) >> 20) & 0x7ffu) + 45u <
         (((unsigned)__double2hiint(diag) >> 20) & 0x7ffu);
}
__device__ __forceinline__ bool no_pivot(double piv, double diag) {
  return !(piv != 0.0) || !isfinite(piv) || cancels(piv, diag);
}

// LU of one block without pivoting and (-T)^{-1} by substitution, in place in
// global memory, by a CTA: rare, so that only the call costs the kernels above
// registers.  The pivot test of the set-up.
__device__ __noinline__ void plain_block(const double* T, double* lu, double* ninv, int2* eninv,
                                         int m, Header* hdr) {
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int e = tid; e < m * m; e += nt) {
    lu[e] = T[e];
    ninv[e] = e % m == e / m ? -1.0 : 0.0;
  }
  __syncthreads();
  for (int k = 0; k < m; ++k) {
    const double piv = lu[k * m + k];
    if (!(piv != 0.0) || !isfinite(piv)) {
      if (tid == 0) latch(hdr, MC_ERR_SINGULAR_BLOCK);
      return;
    }
    const int n = m - k - 1;
    for (int i = k + 1 + tid; i < m; i += nt) lu[k * m + i] = lu[k * m + i] / piv;
    __syncthreads();
    for (int e = tid; e < n * n; e += nt) {
      const int i = k + 1 + e % n, j = k + 1 + e / n;
      lu[j * m + i] = fma(-lu[k * m + i], lu[j * m + k], lu[j * m + i]);
    }
    __syncthreads();
  }
  for (int k = 0; k < m; ++k) {   // L^{-1}
    const int n = m - k - 1;
    for (int e = tid; e < n * m; e += nt) {
      const int i = k + 1 + e % n, c = e / n;
      ninv[c * m + i] = fma(-lu[k * m + i], ninv[c * m + k], ninv[c * m + i]);
    }
    __syncthreads();
  }
  for (int k = m - 1; k >= 0; --k) {   // U^{-1}
    for (int c = tid; c < m; c += nt) ninv[c * m + k] = ninv[c * m + k] / lu[k * m + k];
    __syncthreads();
    for (int e = tid; e < k * m; e += nt) {
      const int i = e % k, c = e / k;
      ninv[c * m + i] = fma(-lu[k * m + i], ninv[c * m + k], ninv[c * m + i]);
    }
    __syncthreads();
  }
  Exps x;
  for (int e = tid; e < m * m; e += nt) {
    const double v = ninv[e] + 0.0;   // no -0
    ninv[e] = v;
    x.take(v);
  }
  x.join(eninv, (tid & 31) == 0);
}

template <int G, int R>
__device__ __forceinline__ void gj_update(double (&A)[R][R], const double* row, const double* cs,
                                          int ti, int tj, int kb, bool own_row, bool own_col) {
  double c[R], r[R];
#pragma unroll
  for (int a = 0; a < R; ++a) {
    c[a] = cs[ti + G * a];
    r[a] = row[tj + G * a];
  }
#pragma unroll
  for (int b = 0; b < R; ++b)
    if (b == kb && own_col) {
      r[b] = 1.0;
#pragma unroll
      for (int a = 0; a < R; ++a) A[a][b] = 0.0;
    }
#pragma unroll
  for (int a = 0; a < R; ++a)
    if (a == kb && own_row) {
#pragma unroll
      for (int b = 0; b < R; ++b) A[a][b] = 0.0;
    }
#pragma unroll
  for (int a = 0; a < R; ++a)
#pragma unroll
    for (int b = 0; b < R; ++b) A[a][b] = fma(-c[a], r[b], A[a][b]);
#pragma unroll
  for (int a = 0; a < R; ++a)
    if (a == kb && own_row && own_col) A[a][a] = 0.0;   // 1/pivot is kept apart
}

// Blocks of up to 128 rows: G = 16 (one block per CTA) or G = 4 (m <= 16: 16 blocks
// per CTA, half a warp each).
template <int G, int R>
struct GjBlock {
  static constexpr int N = 256 / (G * G), MP = G * R;
  static constexpr int B = R <= 4 ? 3 : R <= 6 ? 2 : 1;   // CTAs per SM
  static size_t doubles(int m) { return ((size_t)6 * MP + (size_t)m * (m + 1) + 1) / 2 * 2; }
};

template <int G, int R>
__global__ void __launch_bounds__(256, GjBlock<G, R>::B) k_gj(const double* __restrict__ tdd,
                                                             double* lu, double* ninv, int2* eninv,
                                                             int64_t L, int m, int ms, int per,
                                                             Header* hdr) {
  extern __shared__ double sm[];
  __shared__ int s_bad[256 / (G * G)];
  constexpr int N = GjBlock<G, R>::N, MP = G * R;
  const int grp = threadIdx.x / (G * G), t = threadIdx.x % (G * G), ti = t % G, tj = t / G;
  double* row = sm + (size_t)grp * per;   // [2][MP]
  double* col = row + 2 * MP;             // [2][MP]
  double* cs = col + 2 * MP;              // [MP]
  double* base = cs + MP;                 // [MP] first part of the diagonal
  double* LU = base + MP;                 // column j at j (m + 1)
  auto sync = []() {
    if constexpr (G == 16)
      __syncthreads();
    else
      __syncwarp();
  };
  for (int64_t l0 = (int64_t)blockIdx.x * N; l0 < L; l0 += (int64_t)gridDim.x * N) {
    const int64_t l = l0 + grp;
    const bool live = l < L;
    double A[R][R];
#pragma unroll
    for (int a = 0; a < R; ++a)
#pragma unroll
      for (int b = 0; b < R; ++b) {
        const int i = ti + G * a, j = tj + G * b;
        A[a][b] = live && i < m && j < m ? tdd[(size_t)l * ms + (size_t)j * m + i]
                                         : (i == j ? 1.0 : 0.0);
        if (a == b && ti == tj) {
          base[i] = A[a][b];
          A[a][b] = 0.0;
        }
      }
    if (ti == 0)
#pragma unroll
      for (int b = 0; b < R; ++b) row[tj + G * b] = A[0][b];
    if (tj == 0)
#pragma unroll
      for (int a = 0; a < R; ++a) col[ti + G * a] = A[a][0];
    if (t == 0) s_bad[grp] = 0;
    sync();
    bool bad = false;
#pragma unroll
    for (int kb = 0; kb < R; ++kb) {
#pragma unroll 1
      for (int kk = 0; kk < G; ++kk) {
        const int k = kb * G + kk;
        if (k >= m || (G == 16 && bad)) break;
        const double* rw = row + (k & 1) * MP;
        const double* cl = col + (k & 1) * MP;
        if (G != 16 || (threadIdx.x >> 5) == (k & 7)) {
          const double piv = base[k] + rw[k];
          const double p = 1.0 / piv;
          for (int i = G == 16 ? (int)(threadIdx.x & 31) : t; i < m; i += G == 16 ? 32 : G * G) {
            const double c = cl[i] * p;
            cs[i] = i == k ? -p : c;
            if (i > k) LU[k * (m + 1) + i] = c;
            if (i >= k) LU[i * (m + 1) + k] = i == k ? piv : rw[i];
          }
          if (G != 16 && no_pivot(piv, base[k])) s_bad[grp] = 1;
        } else if (threadIdx.x == 32 * ((k + 1) & 7)) {   // another warp, not on the critical path
          if (no_pivot(base[k] + rw[k], base[k])) s_bad[grp] = 1;
        }
        sync();
        bad = s_bad[grp] != 0;
        if (ti == kk && tj == kk) base[k] = -cs[k];
        gj_update<G, R>(A, rw, cs, ti, tj, kb, ti == kk, tj == kk);
        double* rn = row + ((k + 1) & 1) * MP;
        double* cn = col + ((k + 1) & 1) * MP;
        const bool step = kk == G - 1;   // row k + 1 lies in the next register block
        constexpr int R1 = R - 1;
        const int nk = step ? 0 : kk + 1;
        if (ti == nk)
#pragma unroll
          for (int b = 0; b < R; ++b)
            rn[tj + G * b] = step ? A[kb < R1 ? kb + 1 : kb][b] : A[kb][b];
        if (tj == nk)
#pragma unroll
          for (int a = 0; a < R; ++a)
            cn[ti + G * a] = step ? A[a][kb < R1 ? kb + 1 : kb] : A[a][kb];
        sync();
      }
    }
    if (live && !bad) {
      Exps x;
#pragma unroll
      for (int a = 0; a < R; ++a)
#pragma unroll
        for (int b = 0; b < R; ++b) {
          const int i = ti + G * a, j = tj + G * b;
          if (i < m && j < m) {
            // 0 - x: no -0, whose sign bit would read as negative
            const double v = (i == j ? -base[i] : 0.0) - A[a][b];
            ninv[(size_t)l * ms + (size_t)j * m + i] = v;
            x.take(v);
          }
        }
      x.join(eninv + l, (threadIdx.x & (G == 16 ? 31 : 15)) == 0,
             G == 16 ? 0xffffffffu : 0xffffu << (threadIdx.x & 16));
      for (int j = tj; j < m; j += G)
        for (int i = ti; i < m; i += G)
          lu[(size_t)l * ms + (size_t)j * m + i] = LU[j * (m + 1) + i];
    }
    if (__syncthreads_or(live && bad)) {   // (also: the buffers are rewritten for the next block)
      for (int g = 0; g < N; ++g)
        if (s_bad[g] != 0 && l0 + g < L) {
          const size_t o = (size_t)(l0 + g) * ms;
          plain_block(tdd + o, lu + o, ninv + o, eninv + l0 + g, m, hdr);
        }
      __syncthreads();   // s_bad is cleared for the next block
    }
  }
}

// Blocks of 129 to 256 rows: a cluster of 2 x 2 CTAs, a 32 x 32 grid of threads
// with R x R entries each (512 KB of the four SMs' registers at m = 256).  Row k
// and column k go into the shared memory of the CTAs that need them; one cluster
// barrier a step.  512 blocks of 256: 33.7 -> 21 ms (13.7 at the pipe's rate; a
// step waits for the pivot and the barrier, and 36 clusters run at once).
template <int R>
struct GjBig {
  static constexpr int H = 16 * R;   // a CTA's rows and columns
  static constexpr size_t doubles = 6 * H + 2 + (size_t)H * (H + 1);
};

template <int R>
__global__ void __cluster_dims__(4, 1, 1) __launch_bounds__(256, 1)
    k_gj_cluster(const double* __restrict__ tdd, double* lu, double* ninv, int2* eninv, int64_t L,
                 int m, int ms, Header* hdr) {
  extern __shared__ double sm[];
  constexpr int H = GjBig<R>::H;
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), cr = rank & 1, cc = rank >> 1;
  const int ti = threadIdx.x % 16, tj = threadIdx.x / 16;
  double* row = sm;              // [2][H]: row k at this CTA's columns
  double* col = row + 2 * H;     // [2][H]: column k at this CTA's rows
  double* cs = col + 2 * H;      // [H]
  double* base = cs + H;         // [H] first part of the diagonal (cr == cc)
  double* piv = base + H;        // [2]
  double* LU = piv + 2;          // local column lj at lj (H + 1)
  double* row_peer = cl.map_shared_rank(row, rank ^ 1);   // the other rows, same columns
  double* col_peer = cl.map_shared_rank(col, rank ^ 2);   // the other columns, same rows
  const int i0 = ti + 16 * cr, j0 = tj + 16 * cc;   // entries (i0 + 32 a, j0 + 32 b)
  for (int64_t l = blockIdx.x / 4; l < L; l += gridDim.x / 4) {
    const double* T = tdd + (size_t)l * ms;
    double A[R][R];
#pragma unroll
    for (int a = 0; a < R; ++a)
#pragma unroll
      for (int b = 0; b < R; ++b) {
        const int i = i0 + 32 * a, j = j0 + 32 * b;
        A[a][b] = i < m && j < m ? T[(size_t)j * m + i] : (i == j ? 1.0 : 0.0);
        if (a == b && i0 == j0) {
          base[ti + 16 * a] = A[a][b];
          A[a][b] = 0.0;
        }
      }
    // put row and column k = 32 q + s (s < 32) into buffer f, q a register block
    auto publish = [&](int q, int s, int f) {
      if (cr == (s >> 4) && ti == (s & 15)) {
#pragma unroll
        for (int a = 0; a < R; ++a)
          if (a == q) {
#pragma unroll
            for (int b = 0; b < R; ++b) {
              row[f * H + tj + 16 * b] = A[a][b];
              row_peer[f * H + tj + 16 * b] = A[a][b];
            }
          }
      }
      if (cc == (s >> 4) && tj == (s & 15)) {
#pragma unroll
        for (int b = 0; b < R; ++b)
          if (b == q) {
#pragma unroll
            for (int a = 0; a < R; ++a) {
              col[f * H + ti + 16 * a] = A[a][b];
              col_peer[f * H + ti + 16 * a] = A[a][b];
              if (a == q && cr == (s >> 4) && ti == (s & 15)) {
                const double d = base[ti + 16 * a], v = d + A[a][b];
                for (int p = 0; p < 4; ++p)
                  cl.map_shared_rank(piv, p)[f] = cancels(v, d) ? 0.0 : v;
              }
            }
          }
      }
    };
    publish(0, 0, 0);
    cl.sync();
    bool bad = false;
#pragma unroll
    for (int kb = 0; kb < R; ++kb) {
#pragma unroll 1
      for (int kk = 0; kk < 32; ++kk) {
        const int k = kb * 32 + kk, f = k & 1;
        if (k >= m || bad) break;
        const double pv = piv[f];
        bad = !(pv != 0.0) || !isfinite(pv);   // the same in every CTA
        if (bad) break;
        const bool my_row = cr == (kk >> 4), my_col = cc == (kk >> 4);
        const int lk = (kk & 15) + 16 * kb;    // local index of row / column k
        if ((threadIdx.x >> 5) == (k & 7)) {
          const double p = 1.0 / pv;
          for (int q = threadIdx.x & 31; q < H; q += 32) {
            const int gi = (q & 15) + 16 * cr + 32 * (q >> 4);   // global row of local row q
            const int gj = (q & 15) + 16 * cc + 32 * (q >> 4);
            const double c = col[f * H + q] * p;
            cs[q] = gi == k ? -p : c;
            if (my_col && gi > k) LU[lk * (H + 1) + q] = c;
            if (my_row && gj >= k) LU[q * (H + 1) + lk] = gj == k ? pv : row[f * H + q];
          }
        }
        __syncthreads();
        if (my_row && my_col && ti == (kk & 15) && tj == (kk & 15)) base[lk] = -cs[lk];
        gj_update<16, R>(A, row + f * H, cs, ti, tj, kb, my_row && ti == (kk & 15),
                              my_col && tj == (kk & 15));
        if (k + 1 < m) {
          if (kk == 31)
            publish(kb + 1, 0, f ^ 1);
          else
            publish(kb, kk + 1, f ^ 1);
        }
        cl.sync();
      }
    }
    if (bad) {
      const size_t o = (size_t)l * ms;
      if (rank == 0) plain_block(tdd + o, lu + o, ninv + o, eninv + l, m, hdr);
    } else {
      Exps x;
#pragma unroll
      for (int a = 0; a < R; ++a)
#pragma unroll
        for (int b = 0; b < R; ++b) {
          const int i = i0 + 32 * a, j = j0 + 32 * b;
          if (i < m && j < m) {
            const double v = (i == j ? -base[ti + 16 * a] : 0.0) - A[a][b];
            ninv[(size_t)l * ms + (size_t)j * m + i] = v;
            lu[(size_t)l * ms + (size_t)j * m + i] = LU[(tj + 16 * b) * (H + 1) + ti + 16 * a];
            x.take(v);
          }
        }
      x.join(eninv + l, (threadIdx.x & 31) == 0);
    }
    cl.sync();   // the buffers are rewritten for the next block
  }
}

// ---- coupled operators -------------------------------------------------------
// W = NINV * T for T in {TLO, TUP} (column-major): tiles of 16 RT x 16 RT by 256
// threads with up to RT x RT entries each (fewer in the last tiles of a block),
// panels of 16 columns of NINV staged in shared memory with the 16 rows of T that
// meet them.  FP64-pipe bound, so half of a
// thread's entries are formed on the integer pipes where both blocks allow it
// (fixed_dev.cuh: exact products, one rounding per entry), the others by FP64
// multiply-adds; an entry outside the fixed-point window is formed again in
// FP64.  8192 blocks of 64: 8.6 -> 4.5 ms (6.8 at the FP64 pipe's rate); 512 of
// 256: 82.7 -> 17.4 ms (27).
constexpr int kPanel = 16;   // columns of NINV per panel
template <int TILE>
struct CoupledShared {
  double A[kPanel][TILE];
  double B[kPanel][TILE + 1];
  uint64_t X[kPanel][TILE + 1];   // integer form of B
};

// One tile: rows i0 + ti + 16 a (a < RA), columns j0 + tj + 16 b (b < RB) of W.
template <int TILE, int RA, int RB, bool FIX>
__device__ __forceinline__ Exps coupled_tile(CoupledShared<TILE>& sh, const double* Nl,
                                                 const double* T, double* W, int etot, int i0,
                                                 int j0, int m) {
  using namespace dev;
  constexpr int RF = FIX ? RB / 2 : 0, RX = RF > 0 ? RF : 1;   // columns on the integer pipes
  const int ti = threadIdx.x % 16, tj = threadIdx.x / 16;
  double acc[RA][RB];
  uint32_t fa[RA][RX][4], seen[RA][RX];
#pragma unroll
  for (int a = 0; a < RA; ++a) {
#pragma unroll
    for (int b = 0; b < RB; ++b) acc[a][b] = 0.0;
#pragma unroll
    for (int b = 0; b < RX; ++b) {
      fa[a][b][0] = fa[a][b][1] = fa[a][b][2] = fa[a][b][3] = 0u;
      seen[a][b] = 0u;
    }
  }
  for (int k0 = 0; k0 < m; k0 += kPanel) {
    __syncthreads();
    for (int e = threadIdx.x; e < kPanel * 16 * RA; e += 256) {
      const int k = e / (16 * RA), i = e % (16 * RA);
      sh.A[k][i] = k0 + k < m && i0 + i < m ? Nl[(size_t)(k0 + k) * m + i0 + i] : 0.0;
    }
    for (int e = threadIdx.x; e < kPanel * 16 * RB; e += 256) {
      const int k = e % kPanel, j = e / kPanel;
      const double v = k0 + k < m && j0 + j < m ? T[(size_t)(j0 + j) * m + k0 + k] : 0.0;
      sh.B[k][j] = v;
      if (RF > 0) sh.X[k][j] = fixed_entry(v);
    }
    __syncthreads();
#pragma unroll 2
    for (int k = 0; k < kPanel; ++k) {
      double a[RA];
#pragma unroll
      for (int q = 0; q < RA; ++q) a[q] = sh.A[k][ti + 16 * q];
#pragma unroll
      for (int b = 0; b < RB; ++b) {
        if (b < RF) {
          const uint64_t x = sh.X[k][tj + 16 * b];
          const uint32_t xl = (uint32_t)x & 0xfffff800u, xh = (uint32_t)(x >> 32);
          const int s = etot - (int)((uint32_t)x & 0x7ffu);
#pragma unroll
          for (int q = 0; q < RA; ++q)
            fixed_fma(fa[q][b < RF ? b : 0], a[q], xl, xh, s, &seen[q][b < RF ? b : 0]);
        } else {
          const double v = sh.B[k][tj + 16 * b];
#pragma unroll
          for (int q = 0; q < RA; ++q) acc[q][b] = fma(a[q], v, acc[q][b]);
        }
      }
    }
  }
  Exps e;
#pragma unroll
  for (int b = 0; b < RB; ++b)
#pragma unroll
    for (int a = 0; a < RA; ++a) {
      const int i = i0 + ti + 16 * a, j = j0 + tj + 16 * b;
      if (i >= m || j >= m) continue;
      double v = acc[a][b];
      if (b < RF) {
        bool bad = false;
        v = fixed_value(fa[a][b < RF ? b : 0], seen[a][b < RF ? b : 0], etot, bad);
        if (bad) {
          v = 0.0;
          for (int k = 0; k < m; ++k) v = fma(Nl[(size_t)k * m + i], T[(size_t)j * m + k], v);
        }
      }
      W[(size_t)j * m + i] = v;
      e.take(v);
    }
  return e;
}

// 16-row groups of a tile that starts at x, rounded up to a size that has code.
__device__ __forceinline__ int tile_groups(int x, int m) {
  const int g = (m - x + 15) / 16;
  return g >= 3 ? 4 : g;
}

template <int RT>
__global__ void __launch_bounds__(256, 2) k_coupled(const double* __restrict__ ninv,
                                                    const double* __restrict__ tlo,
                                                    const double* __restrict__ tup,
                                                    double* __restrict__ wlo,
                                                    double* __restrict__ wup, const int2* en,
                                                    const int2* elo, const int2* eup, int2* ewlo,
                                                    int2* ewup, int64_t L, int m, int ms,
                                                    int tiles) {
  constexpr int TILE = 16 * RT;
  __shared__ CoupledShared<TILE> sh;
  const int64_t total = L * 2 * tiles * tiles;
  for (int64_t w = blockIdx.x; w < total; w += gridDim.x) {
    // tile by tile over all levels: every CTA gets its share of full and partial tiles
    const int tile = (int)(w / (2 * L));
    const int64_t rest = w - tile * 2 * L, l = rest >> 1;
    const int h = (int)(rest & 1);
    const int i0 = (tile % tiles) * TILE, j0 = (tile / tiles) * TILE;
    const double* Nl = ninv + (size_t)l * ms;
    const double* T = (h == 0 ? tlo : tup) + (size_t)l * ms;
    double* W = (h == 0 ? wlo : wup) + (size_t)l * ms;
    const int ea = en[l].x, eb = (h == 0 ? elo : eup)[l].x, etot = ea + eb;
    const bool fix = dev::fixed_ok(ea) && dev::fixed_ok(eb);
    Exps e;
    auto run = [&](auto ra, auto rb) {
      constexpr int RA = decltype(ra)::value, RB = decltype(rb)::value;
      if constexpr (RA <= RT && RB <= RT)
        e = fix && RB > 1 ? coupled_tile<TILE, RA, RB, (RB > 1)>(sh, Nl, T, W, etot, i0, j0, m)
                          : coupled_tile<TILE, RA, RB, false>(sh, Nl, T, W, etot, i0, j0, m);
    };
    using I1 = std::integral_constant<int, 1>;
    using I2 = std::integral_constant<int, 2>;
    using I4 = std::integral_constant<int, 4>;
    switch (tile_groups(i0, m) * 8 + tile_groups(j0, m)) {
      case 9: run(I1(), I1()); break;
      case 10: run(I1(), I2()); break;
      case 12: run(I1(), I4()); break;
      case 17: run(I2(), I1()); break;
      case 18: run(I2(), I2()); break;
      case 20: run(I2(), I4()); break;
      case 33: run(I4(), I1()); break;
      case 34: run(I4(), I2()); break;
      default: run(I4(), I4()); break;
    }
    e.join((h == 0 ? ewlo : ewup) + l, (threadIdx.x & 31) == 0);
  }
}

// W for m <= 16: one entry per thread over all blocks (the sweeps of such blocks
// use no exponents).
__global__ void __launch_bounds__(256) k_coupled_small(const double* __restrict__ ninv,
                                                       const double* __restrict__ tlo,
                                                       const double* __restrict__ tup,
                                                       double* __restrict__ wlo,
                                                       double* __restrict__ wup, int64_t L, int m,
                                                       int ms) {
  const int mm = m * m;
  const int64_t total = 2 * L * mm;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = t / mm, l = b >> 1;
    const int e = (int)(t - b * mm), j = e / m, i = e - j * m;
    const double* N = ninv + (size_t)l * ms + i;
    const double* T = ((b & 1) ? tup : tlo) + (size_t)l * ms + j * m;
    double acc = 0.0;
#pragma unroll 4
    for (int k = 0; k < m; ++k) acc = fma(N[k * m], T[k], acc);
    ((b & 1) ? wup : wlo)[(size_t)l * ms + e] = acc;
  }
}

// Zero quadrants of a paired pentadiagonal chain (column-major blocks):
// TLO rows h.. of columns ..h and TUP rows ..h of columns h.., h = m/2.
__global__ void k_check_paired(const double* __restrict__ tlo, const double* __restrict__ tup,
                               int64_t L, int m, int ms, Header* hdr) {
  const int h = m / 2;
  const int64_t per = (int64_t)h * h;
  const int64_t total = L * per;
  bool bad = false;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t l = t / per, e = t % per;
    const int a = (int)(e / h), b = (int)(e % h);   // column a, row b of the quadrant
    bad |= tlo[(size_t)l * ms + (size_t)a * m + h + b] != 0.0;
    bad |= tup[(size_t)l * ms + (size_t)(h + a) * m + b] != 0.0;
  }
  if (bad) latch(hdr, MC_ERR_ARG);
}

__global__ void __launch_bounds__(256) k_layout_diag(const double* diag, int d, double* plane,
                                                     int2* bexp, int64_t L, int m, int ms) {
  const int64_t mm = (int64_t)m * m;
  const int chunks = (ms + kChunk - 1) / kChunk, lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < L * chunks;
       t += nw) {
    const int64_t l = t / chunks, k = l + d;
    Exps x = copy_chunk(k >= 0 && k < L ? diag + k * mm : nullptr, plane + (size_t)l * ms,
                        (int)(t - l * chunks) * kChunk, (int)mm, ms, lane);
    x.join(bexp + l, lane == 0);
  }
}

// block_exp (but for the rows) of TLO and TUP where the blocks did not come through k_layout.
__global__ void __launch_bounds__(256) k_block_exp(const double* __restrict__ tlo,
                                                   const double* __restrict__ tup, int2* elo,
                                                   int2* eup, int64_t L, int m, int ms) {
  const int chunks = (ms + kChunk - 1) / kChunk, lane = threadIdx.x & 31;
  const int64_t total = 2 * L * chunks, nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < total; t += nw) {
    const int64_t b = t / chunks, l = b >> 1;
    const int e0 = (int)(t - b * chunks) * kChunk, e1 = min(e0 + kChunk, m * m);
    const double* p = ((b & 1) ? tup : tlo) + (size_t)l * ms;
    Exps x;
    for (int i = e0 + lane; i < e1; i += 32) x.take(__ldcs(p + i));
    x.join(((b & 1) ? eup : elo) + l, lane == 0);
  }
}

// The rows' part of block_exp: the smallest over the rows (that are not zero) of a
// row's largest entry.  Local blocks whose phases form a long line have inverses
// whose entries span hundreds of bits with every row's largest at the same size.
// Blocks that span up to 2^16 are left at their smallest entry, which loses little
// there, and are not read again; a warp per other block.
struct WeakRows {
  int n;
  const double* plane[3 + kMaxFar];
  int2* exps[3 + kMaxFar];
};
__global__ void __launch_bounds__(256) k_weak_rows(WeakRows p, int64_t L, int m, int ms) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < p.n * L; t += nw) {
    const int64_t l = t % L;
    const int k = (int)(t / L);
    int2* to = p.exps[k] + l;
    const int2 e = *to;
    if (e.x >= 2047 || e.x + e.y <= 4096 + 16) continue;   // (no entries: 0 + 0)
    const double* M = p.plane[k] + (size_t)l * ms;
    unsigned weak = 0u;
    for (int r0 = 0; r0 < m; r0 += 32) {
      const int row = r0 + lane;
      unsigned most = 0u;
      bool any = false;
      if (row < m)
        for (int j = 0; j < m; ++j) {
          const double v = M[(size_t)j * m + row];
          any = any || !dev::is_zero(v);
          most = max(most, dev::exp_field(v));
        }
      if (any) weak = max(weak, 4096u - most);
    }
    weak = __reduce_max_sync(0xffffffffu, weak);
    if (lane == 0) to->y = (int)(weak << 16) | (e.y & 0xffff);
  }
}

int copy_blocks(int64_t warps) {
  const int64_t nb = (warps + 7) / 8;
  return (int)(nb < 4096 ? nb : 4096);
}

}  // namespace

cudaError_t launch_weak_rows(const double* planes, int2* bexp, const Layout& y, int coupled,
                             cudaStream_t s) {
  const size_t pe = y.plane_bytes / sizeof(double);
  WeakRows p{};
  auto add = [&](int k) {
    p.plane[p.n] = planes + (size_t)k * pe;
    p.exps[p.n++] = bexp + (size_t)k * y.L;
  };
  add(coupled ? kPlaneWLO : kPlaneTLO);
  add(coupled ? kPlaneWUP : kPlaneTUP);
  if (!coupled) add(kPlaneNINV);
  for (int j = 0; j < y.nfar; ++j) add(y.far_base + j);
  k_weak_rows<<<copy_blocks(p.n * y.L), 256, 0, s>>>(p, y.L, y.m, y.ms);
  return cudaGetLastError();
}

cudaError_t launch_block_exp(const double* planes, int2* bexp, const Layout& y, cudaStream_t s) {
  const size_t pe = y.plane_bytes / sizeof(double);
  const int chunks = (y.ms + kChunk - 1) / kChunk;
  k_block_exp<<<copy_blocks(2 * y.L * chunks), 256, 0, s>>>(
      planes + kPlaneTLO * pe, planes + kPlaneTUP * pe, bexp + kPlaneTLO * y.L,
      bexp + kPlaneTUP * y.L, y.L, y.m, y.ms);
  return cudaGetLastError();
}

cudaError_t launch_layout_diag(const double* diag, int d, double* plane, int2* bexp,
                               const Layout& lay, cudaStream_t s) {
  const int chunks = (lay.ms + kChunk - 1) / kChunk;
  k_layout_diag<<<copy_blocks(lay.L * chunks), 256, 0, s>>>(diag, d, plane, bexp, lay.L, lay.m,
                                                            lay.ms);
  return cudaGetLastError();
}

cudaError_t launch_check_paired(const double* tlo, const double* tup, const Layout& lay,
                                Header* hdr, cudaStream_t s) {
  k_check_paired<<<1024, 256, 0, s>>>(tlo, tup, lay.L, lay.m, lay.ms, hdr);
  return cudaGetLastError();
}

cudaError_t launch_layout(const double* dn, const double* loc, const double* up, double* planes,
                          int2* bexp, const Layout& lay, cudaStream_t s) {
  const size_t pe = lay.plane_bytes / sizeof(double);
  const int chunks = (lay.ms + kChunk - 1) / kChunk;
  k_layout<<<copy_blocks(3 * lay.L * chunks), 256, 0, s>>>(
      dn, loc, up, planes + kPlaneTLO * pe, planes + kPlaneTUP * pe, planes + kPlaneTDD * pe,
      bexp + kPlaneTLO * lay.L, bexp + kPlaneTUP * lay.L, lay.L, lay.m, lay.ms);
  return cudaGetLastError();
}

namespace {

struct FactorArgs {
  const double* tdd;
  double *lu, *ninv;
  int2* eninv;
  int64_t L;
  int m, ms, sms;
  Header* hdr;
};

template <int G, int R>
cudaError_t gj(const FactorArgs& f, cudaStream_t s) {
  constexpr int N = GjBlock<G, R>::N;
  const size_t per = GjBlock<G, R>::doubles(f.m), bytes = N * per * sizeof(double);
  const cudaError_t e = cudaFuncSetAttribute(
      k_gj<G, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  int occ = 0;   // every CTA resident: the blocks are dealt out once
  const cudaError_t e2 =
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_gj<G, R>, 256, bytes);
  if (e2 != cudaSuccess) return e2;
  int64_t nb = (f.L + N - 1) / N;
  if (nb > (int64_t)occ * f.sms) nb = (int64_t)(occ < 1 ? 1 : occ) * f.sms;
  k_gj<G, R><<<(int)nb, 256, bytes, s>>>(f.tdd, f.lu, f.ninv, f.eninv, f.L, f.m, f.ms, (int)per,
                                         f.hdr);
  return cudaGetLastError();
}

template <int R>
cudaError_t gj_big(const FactorArgs& f, cudaStream_t s) {
  const size_t bytes = GjBig<R>::doubles * sizeof(double);
  const cudaError_t e = cudaFuncSetAttribute(
      k_gj_cluster<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  // as many clusters as run at once (the SMs of a GPC that are left over from
  // clusters of four stay idle: 36 of the 38 that the SM count suggests), so
  // that none waits for a whole block's time
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(4 * (unsigned)(f.sms / 4 < 1 ? 1 : f.sms / 4));
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = bytes;
  int fit = 0;
  const cudaError_t e2 =
      cudaOccupancyMaxActiveClusters(&fit, (const void*)k_gj_cluster<R>, &cfg);
  if (e2 != cudaSuccess) return e2;
  int64_t nc = fit < 1 ? 1 : fit;
  if (nc > f.L) nc = f.L;
  k_gj_cluster<R><<<(int)(4 * nc), 256, bytes, s>>>(f.tdd, f.lu, f.ninv, f.eninv, f.L, f.m, f.ms,
                                                    f.hdr);
  return cudaGetLastError();
}

cudaError_t gj_dispatch(const FactorArgs& f, cudaStream_t s) {
  if (f.m <= 8) return gj<4, 2>(f, s);
  if (f.m <= 16) return gj<4, 4>(f, s);
  if (f.m <= 128) switch ((f.m + 15) / 16) {
      case 2: return gj<16, 2>(f, s);
      case 3: return gj<16, 3>(f, s);
      case 4: return gj<16, 4>(f, s);
      case 5: return gj<16, 5>(f, s);
      case 6: return gj<16, 6>(f, s);
      case 7: return gj<16, 7>(f, s);
      default: return gj<16, 8>(f, s);
    }
  switch ((f.m + 31) / 32) {
    case 5: return gj_big<5>(f, s);
    case 6: return gj_big<6>(f, s);
    case 7: return gj_big<7>(f, s);
    default: return gj_big<8>(f, s);
  }
}

}  // namespace

cudaError_t launch_factor(double* planes, int2* bexp, const Layout& lay, Header* hdr, int coupled,
                          int num_sms, cudaStream_t s) {
  const size_t pe = lay.plane_bytes / sizeof(double);
  const int m = lay.m;
  const int64_t L = lay.L;
  const FactorArgs f{planes + kPlaneTDD * pe, planes + kPlaneLU * pe, planes + kPlaneNINV * pe,
                     bexp + kPlaneNINV * L, L, m, lay.ms, num_sms, hdr};
  const cudaError_t e = gj_dispatch(f, s);
  if (e != cudaSuccess || !coupled) return e;
  if (m <= 16) {
    const int64_t nb = (2 * L * m * m + 255) / 256;
    k_coupled_small<<<(int)(nb < 8192 ? nb : 8192), 256, 0, s>>>(
        planes + kPlaneNINV * pe, planes + kPlaneTLO * pe, planes + kPlaneTUP * pe,
        planes + kPlaneWLO * pe, planes + kPlaneWUP * pe, L, m, lay.ms);
    return cudaGetLastError();
  }
  const int rt = m <= 32 ? 2 : 4, tiles = (m + 16 * rt - 1) / (16 * rt);
  int64_t nb = L * 2 * tiles * tiles;
  if (nb > 2ll * num_sms) nb = 2ll * num_sms;
  auto kernel = rt == 2 ? k_coupled<2> : k_coupled<4>;
  kernel<<<(int)nb, 256, 0, s>>>(planes + kPlaneNINV * pe, planes + kPlaneTLO * pe,
                                 planes + kPlaneTUP * pe, planes + kPlaneWLO * pe,
                                 planes + kPlaneWUP * pe, bexp + kPlaneNINV * L,
                                 bexp + kPlaneTLO * L, bexp + kPlaneTUP * L, bexp + kPlaneWLO * L,
                                 bexp + kPlaneWUP * L, L, m, lay.ms, tiles);
  return cudaGetLastError();
}

}  // namespace mc
