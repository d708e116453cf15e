// Staircase sweeps of a chain that fits the shared memory of one thread-block
// cluster: the operators are loaded once per launch and every half-sweep runs
// between two cluster barriers.
//
// A small chain's sweep through global memory (k_sweeps, k_sweeps_lp) is a
// serial chain of L2 round trips: the wait for the neighbours' counters, their
// acquire, the vectors, each operator block, the fence and the release, 5.3 us
// per half-sweep whatever the arithmetic.  Resident, 64 levels of 8: 10.7 -> 1.29
// us a sweep (coupled 7.9 -> 0.94); 130 levels of 32, as many as fit: 17 -> 9.4;
// 1500 levels of 8: 12.6 -> 7.1 (both FP64 pipe of 16 SMs).  What is left of a
// small sweep is the FP64 pipe's 64 clocks per instruction and warp, 11 of them
// in a row per half-sweep, and about 350 clocks of exchange.
// Here CTA r of the cluster owns a contiguous range of levels, its blocks and
// vectors stay on chip, and the two boundary levels of the range are also pushed
// into the neighbouring CTAs' shared memory (distributed shared memory).  The
// hardware co-schedules a cluster's CTAs, so they may wait for one another.
#pragma once
#include <cooperative_groups.h>
#include <stdint.h>

#include "mc_internal.cuh"
#include "wave_dev.cuh"

namespace mc {
namespace res {

namespace cg = cooperative_groups;

constexpr int kThreads = 256;

__device__ __forceinline__ double elem(double v) { return v; }
__device__ __forceinline__ float elem(float v) { return v; }
__device__ __forceinline__ float elem(unsigned short v) { return __uint_as_float((unsigned)v << 16); }
__device__ __forceinline__ double madd(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float madd(float a, float b, float c) { return fmaf(a, b, c); }

// Elements of a block in shared memory: m^2 rounded up to 16 bytes.
template <typename T>
__host__ __device__ constexpr size_t packed(int m) {
  constexpr size_t e = 16 / sizeof(T);
  return ((size_t)m * m + e - 1) / e * e;
}

// Shared memory of a CTA holding up to `n` levels: operator planes first, then
// vectors with one halo level on either side.
struct Carve {
  size_t a, b, c, x, z, g, total;
};
template <typename T, typename TC, typename V, bool COUPLED>
__host__ __device__ inline Carve carve(int n, int m) {
  auto up = [](size_t v) { return (v + 15) / 16 * 16; };
  Carve k;
  size_t o = 0;
  k.a = o;
  o += n * packed<T>(m) * sizeof(T);
  k.b = o;
  o += n * packed<T>(m) * sizeof(T);
  k.c = o;
  if (!COUPLED) o += n * packed<TC>(m) * sizeof(TC);
  k.x = o;
  o += up((size_t)(n + 2) * m * sizeof(V));
  k.z = o;   // FP64 only: the last sweep's result (x keeps the previous iterate)
  if (sizeof(V) == 8) o += up((size_t)(n + 2) * m * sizeof(V));
  k.g = o;   // inverse mode: T_lo v + T_up v; low precision: q
  o += up((size_t)n * m * sizeof(V) * (COUPLED || sizeof(V) == 8 ? 1 : 2));
  k.total = o;
  return k;
}

// Range of levels of CTA r of C.
__host__ __device__ inline int range_begin(int L, int C, int r) {
  const int base = L / C, rem = L % C;
  return r * base + (r < rem ? r : rem);
}

// How the threads cover the rows of a half-sweep's levels.  With enough rows a
// thread owns one row of one level (rows of consecutive levels flattened, so no
// lane idles whatever m is).  With few rows of m <= 16, groups of mp S lanes
// share a level, mp = m rounded up to a power of two, S lanes of each row taking
// every S-th column (partial sums added by shuffles): this shortens the serial
// chain of multiply-adds (64 clocks each in FP64) and no more warps than needed
// issue FP64 instructions (16 clocks of the SM's pipe each, whatever the lanes
// in use).
struct Cover {
  int mp, S, gs;   // S = 1: flattened rows; else gs = mp S lanes per level
};
__device__ __forceinline__ Cover cover(int m, int n_half) {
  Cover c{1, 1, 1};
  if (m > 16) return c;
  while (c.mp < m) c.mp *= 2;
  while (c.mp * c.S < 32 && c.S < m && n_half * c.mp * c.S * 2 <= kThreads) c.S *= 2;
  c.gs = c.mp * c.S;
  return c;
}

// sum_j A(i, j) p_j sa + B(i, j) q_j sb over this thread's columns.  (FP64: one
// chain, a warp's FP64 instructions issue 64 clocks apart anyway.)
template <typename T, typename V>
__device__ __forceinline__ V dot2(const T* A, const T* B, const V* p, const V* q, int m, int i,
                                  int j0, int S, V sa, V sb) {
  V a = 0, b = 0;
  const T *pa = A + j0 * m + i, *pb = B + j0 * m + i;
#pragma unroll 4
  for (int j = j0; j < m; j += S, pa += S * m, pb += S * m) {
    a = madd(elem(*pa), p[j], a);
    if constexpr (sizeof(V) == 8)
      a = madd(elem(*pb), q[j], a);
    else
      b = madd(elem(*pb), q[j], b);
  }
  if constexpr (sizeof(V) == 8) return a;
  return a * sa + b * sb;
}

template <typename T, typename V>
__device__ __forceinline__ V dot1(const T* A, const V* p, int m, int i, int j0, int S) {
  V a = 0;
  const T* pa = A + j0 * m + i;
#pragma unroll 4
  for (int j = j0; j < m; j += S, pa += S * m) a = madd(elem(*pa), p[j], a);
  return a;
}

// value(u, i, j0, S) per (level u of the half-sweep's n_half, row i), summed
// over the S lanes that share a row, then store(u, i, value).  Warps without
// rows issue nothing.
template <typename V, typename F, typename G>
__device__ __forceinline__ void for_rows(const Cover& c, int m, int n_half, F value, G store) {
  if (c.S == 1) {
    const int rows = n_half * m;
    for (int t = threadIdx.x; t < rows; t += kThreads) {
      const int u = t / m, i = t - u * m;
      store(u, i, value(u, i, 0, 1));
    }
  } else {
    const int i = threadIdx.x & (c.mp - 1), s = (threadIdx.x & (c.gs - 1)) / c.mp;
    const int per = kThreads / c.gs;
    for (int u0 = (threadIdx.x & ~31) / c.gs; u0 < n_half; u0 += per) {   // warp-uniform
      const int u = u0 + (threadIdx.x & 31) / c.gs;
      const bool ok = u < n_half && i < m;
      V v = ok ? value(u, i, s, c.S) : V(0);
      for (int o = c.mp; o < c.gs; o *= 2) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (ok && s == 0) store(u, i, v);
    }
  }
}

// Operators and vectors of a chain (or of one request of a batch).
template <typename T, typename TC, typename V>
struct Chain {
  const T* A;
  const T* B;
  const TC* C;
  int64_t as, cs;        // block strides in elements
  const float* sc;       // low precision: scales of A and B per level
  const V* in;           // start vector (NULL: zero)
  const float* q;        // low precision: right-hand side
  int L, m, par0;
};

// ---- halo exchange -----------------------------------------------------------
// Each boundary level is pushed into the neighbouring CTA's halo with st.async,
// whose bytes complete a phase of that CTA's mbarrier; the neighbour's threads
// that read the halo wait for the phase.  Once per sweep and side: the writer
// can only push the next version after it has received the reader's own
// boundary level, computed after the read, so no slot is overwritten early and
// no barrier counts two phases.  660 clocks a half-sweep for a cluster barrier
// behind a distributed store against about 350 for this and a block barrier.
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint32_t peer_addr(uint32_t a, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ void push(uint32_t dst, uint32_t bar, double v) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(dst),
               "l"(__double_as_longlong(v)), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void push(uint32_t dst, uint32_t bar, float v) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(dst),
               "r"(__float_as_uint(v)), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void bar_init(uint32_t bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void bar_expect(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
// Wait for the completion of the phase of this parity, at most 2 s of the
// global timer (then MC_ERR_TIMEOUT is latched; no wait outlasts a latched
// error, so the launch always ends).
__device__ __forceinline__ void bar_wait(uint32_t bar, uint32_t parity, int* status) {
  unsigned long long t0 = 0;
  for (int it = 0;; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return;
    if (it == 0) {
      t0 = dev::global_ns();
    } else if ((it & 255) == 0) {
      if (*reinterpret_cast<volatile int*>(status) == (int)MC_ERR_TIMEOUT) return;
      if (dev::global_ns() - t0 > 2000000000ull) {
        atomicCAS(status, 0, (int)MC_ERR_TIMEOUT);
        return;
      }
    }
  }
}

// One CTA's side of the exchange.  bar[0] / bar[1]: this CTA's left / right halo;
// rh[side]: the half-sweep that reads it (the one of the boundary level's parity).
struct Halo {
  uint32_t bar[2];                 // own barriers
  uint32_t xl, xr, zl, zr;         // halo slots of the neighbours (x and z)
  uint32_t bl, br;                 // their barriers
  bool left, right;
  int rh[2];
  uint32_t bytes;                  // of one version
  int* status;
};

// Before half-sweep hs of sweep kk reads the left (side 0) or right halo: the
// neighbour has pushed kk versions by then if hs = 0 (the last one in its second
// half of the sweep before), kk + 1 if hs = 1.
__device__ __forceinline__ void halo_wait(const Halo& h, int side, int kk, int hs) {
  const int need = kk + hs;
  if (need > 0 && (side == 0 ? h.left : h.right))
    bar_wait(h.bar[side], (uint32_t)(need - 1) & 1u, h.status);
}

// After that half-sweep's block barrier (its version has been received): arm
// the barrier for the next one.  K versions in all; the first is armed before
// the sweeps.
__device__ __forceinline__ void halo_next(const Halo& h, int kk, int hs, int K) {
  if (threadIdx.x < 2) {
    const int side = threadIdx.x, need = kk + hs;
    if ((side == 0 ? h.left : h.right) && h.rh[side] == hs && need > 0 && need < K)
      bar_expect(h.bar[side], h.bytes);
  }
}

// Chains whose half-sweep gives every thread at most one (level, row, column
// group): the operators' entries stay in registers, CPL columns a lane and
// operator for both parities; the inverse's input moves between the lanes of
// a level by shuffles.
template <typename T, typename TC, typename V, bool COUPLED, int CPL>
__device__ __forceinline__ void sweeps_tiny(const Chain<T, TC, V>& h, int K, const Cover& c, V* x,
                                            V* z, int l0, int n, const Halo& ha) {
  const int L = h.L, m = h.m;
  const int i = threadIdx.x & (c.mp - 1), s = (threadIdx.x & (c.gs - 1)) / c.mp;
  const int u = threadIdx.x / c.gs;
  const int base = (threadIdx.x & 31) & ~(c.gs - 1);   // first lane of the level's group
  V A[2][CPL], B[2][CPL], C[2][CPL], q[2];
  int col[CPL];
#pragma unroll
  for (int k = 0; k < CPL; ++k) {
    const int j = s + c.S * k;
    col[k] = j < m ? j : m - 1;   // entries beyond m are zero
  }
  bool ok[2], busy[2];
  int tt[2];
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int p = e == 0 ? h.par0 : 1 - h.par0;
    const int t0 = (l0 ^ p) & 1, nh = n > t0 ? (n - t0 + 1) / 2 : 0;
    tt[e] = t0 + 2 * (u < nh ? u : 0);
    ok[e] = u < nh && i < m;
    busy[e] = (threadIdx.x & ~31) / c.gs < nh;   // any lane of the warp
    const int64_t l = l0 + tt[e];
    V sa = 1, sb = 1;
    if (sizeof(V) == 4 && ok[e] && h.sc) {
      sa = (V)h.sc[2 * l];
      sb = (V)h.sc[2 * l + 1];
    }
#pragma unroll
    for (int k = 0; k < CPL; ++k) {
      const int j = s + c.S * k;
      const bool in = ok[e] && j < m;
      A[e][k] = in && l > 0 ? elem(h.A[(size_t)l * h.as + (size_t)j * m + i]) * sa : V(0);
      B[e][k] = in && l < L - 1 ? elem(h.B[(size_t)l * h.as + (size_t)j * m + i]) * sb : V(0);
      C[e][k] = !COUPLED && in ? elem(h.C[(size_t)l * h.cs + (size_t)j * m + i]) : V(0);
    }
    q[e] = sizeof(V) == 4 && ok[e] ? (V)h.q[l * m + i] : V(0);
  }
  for (int kk = 0; kk < K; ++kk) {
    const bool last = sizeof(V) == 8 && kk == K - 1;
    V* dst = last ? z : x;
#pragma unroll
    for (int hs = 0; hs < 2; ++hs) {
      const V* src = hs == 0 ? x : dst;
      if (busy[hs]) {
        const int t = tt[hs];
        if (ok[hs] && t == 0) halo_wait(ha, 0, kk, hs);
        if (ok[hs] && t == n - 1) halo_wait(ha, 1, kk, hs);
        const V* lo = src + t * m;
        const V* up = lo + 2 * m;
        // one chain: a warp's FP64 instructions issue 64 clocks apart, so more
        // chains would only add the sum that joins them
        V v = 0;
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
          v = madd(A[hs][k], lo[col[k]], v);
          v = madd(B[hs][k], up[col[k]], v);
        }
        for (int o = c.mp; o < c.gs; o *= 2) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (!COUPLED) {
          V w = 0;
#pragma unroll
          for (int k = 0; k < CPL; ++k)
            w = madd(C[hs][k], __shfl_sync(0xffffffffu, v, base + col[k]), w);
          for (int o = c.mp; o < c.gs; o *= 2) w += __shfl_xor_sync(0xffffffffu, w, o);
          v = w;
        }
        if (ok[hs] && s == 0) {
          if constexpr (sizeof(V) == 4) v += q[hs];
          dst[(t + 1) * m + i] = v;
          if (t == 0 && ha.left) push((last ? ha.zl : ha.xl) + i * (int)sizeof(V), ha.bl, v);
          if (t == n - 1 && ha.right) push((last ? ha.zr : ha.xr) + i * (int)sizeof(V), ha.br, v);
        }
      }
      __syncthreads();
      halo_next(ha, kk, hs, K);
    }
  }
}

// n blocks of a plane (stride gs, 16-byte aligned, padded to 256 bytes) into
// shared memory by all threads, 8 loads of 16 bytes in flight each; block
// `zero` becomes zero.
template <typename T>
__device__ __forceinline__ void load_plane(T* dst, const T* src, int64_t gs, int n, int m,
                                           int zero) {
  constexpr int E = 16 / sizeof(T);
  const int per = (int)(packed<T>(m) / E), total = n * per;
  uint4* d = reinterpret_cast<uint4*>(dst);
  for (int e0 = threadIdx.x; e0 < total; e0 += 8 * kThreads) {
    uint4 v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int e = e0 + i * kThreads, t = e / per;
      v[i] = e < total && t != zero
                 ? *reinterpret_cast<const uint4*>(src + (size_t)t * gs + (size_t)(e - t * per) * E)
                 : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int e = e0 + i * kThreads;
      if (e < total) d[e] = v[i];
    }
  }
}

// K sweeps.  On return z (FP64) / x (low precision) holds the CTA's levels of
// the result and FP64 x the iterate before the last sweep, halos included.
// bars: two mbarriers in shared memory.
template <typename T, typename TC, typename V, bool COUPLED>
__device__ __forceinline__ void sweeps(const Chain<T, TC, V>& h, int K, unsigned char* smem,
                                       unsigned long long* bars, int* status) {
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), r = (int)cl.block_rank();
  const int L = h.L, m = h.m;
  const int ms = (int)packed<T>(m), mc = (int)packed<TC>(m);
  const int l0 = range_begin(L, C, r), n = range_begin(L, C, r + 1) - l0;
  const int nmax = (L + C - 1) / C;
  const Carve k = carve<T, TC, V, COUPLED>(nmax, m);
  T* A = reinterpret_cast<T*>(smem + k.a);
  T* B = reinterpret_cast<T*>(smem + k.b);
  TC* Cp = reinterpret_cast<TC*>(smem + k.c);
  V* x = reinterpret_cast<V*>(smem + k.x);
  V* z = reinterpret_cast<V*>(smem + k.z);
  V* g = reinterpret_cast<V*>(smem + k.g);
  V* qv = g + (COUPLED ? 0 : (size_t)nmax * m);
  const int tid = threadIdx.x;
  const Cover c = cover(m, (nmax + 1) / 2);   // the same in every CTA
  const int cpl = (m + c.S - 1) / c.S;
  const bool tiny = m <= 16 && ((nmax + 1) / 2) * c.gs <= kThreads && cpl <= 8;
  Halo ha{};
  ha.bar[0] = smem_addr(bars);
  ha.bar[1] = smem_addr(bars + 1);
  ha.left = r > 0;
  ha.right = r < C - 1;
  ha.status = status;
  if (ha.left) {
    const int nl = l0 - range_begin(L, C, r - 1);   // the left CTA's right halo
    ha.xl = peer_addr(smem_addr(x + (nl + 1) * m), r - 1);
    ha.zl = peer_addr(smem_addr(z + (nl + 1) * m), r - 1);
    ha.bl = peer_addr(ha.bar[1], r - 1);
  }
  if (ha.right) {
    ha.xr = peer_addr(smem_addr(x), r + 1);
    ha.zr = peer_addr(smem_addr(z), r + 1);
    ha.br = peer_addr(ha.bar[0], r + 1);
  }
  ha.rh[0] = (l0 & 1) == h.par0 ? 0 : 1;
  ha.rh[1] = ((l0 + n - 1) & 1) == h.par0 ? 0 : 1;
  ha.bytes = (uint32_t)(m * sizeof(V));
  if (tid == 0) {
    bar_init(ha.bar[0]);
    bar_init(ha.bar[1]);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (ha.left) bar_expect(ha.bar[0], ha.bytes);
    if (ha.right) bar_expect(ha.bar[1], ha.bytes);
  }
  // operators, blocks packed; blocks that lead out of the chain are zero
  if (!tiny) {
    load_plane(A, h.A + (size_t)l0 * h.as, h.as, n, m, l0 == 0 ? 0 : -1);
    load_plane(B, h.B + (size_t)l0 * h.as, h.as, n, m, l0 + n == L ? n - 1 : -1);
    if (!COUPLED) load_plane(Cp, h.C + (size_t)l0 * h.cs, h.cs, n, m, -1);
  }
  for (int e = tid; e < (n + 2) * m; e += kThreads) {
    const int64_t j = (int64_t)(l0 - 1) * m + e;
    const V v = h.in && j >= 0 && j < (int64_t)L * m ? h.in[j] : V(0);
    x[e] = v;
    if (sizeof(V) == 8) z[e] = V(0);
  }
  if (sizeof(V) == 4 && !tiny)
    for (int e = tid; e < n * m; e += kThreads) qv[e] = (V)h.q[(int64_t)l0 * m + e];
  cl.sync();
  if (tiny) {
    if (cpl <= 1)
      sweeps_tiny<T, TC, V, COUPLED, 1>(h, K, c, x, z, l0, n, ha);
    else if (cpl <= 2)
      sweeps_tiny<T, TC, V, COUPLED, 2>(h, K, c, x, z, l0, n, ha);
    else if (cpl <= 4)
      sweeps_tiny<T, TC, V, COUPLED, 4>(h, K, c, x, z, l0, n, ha);
    else
      sweeps_tiny<T, TC, V, COUPLED, 8>(h, K, c, x, z, l0, n, ha);
  } else {
    for (int kk = 0; kk < K; ++kk) {
      const bool last = sizeof(V) == 8 && kk == K - 1;
      V* dst = last ? z : x;
#pragma unroll 1
      for (int hs = 0; hs < 2; ++hs) {
        const int p = hs == 0 ? h.par0 : 1 - h.par0;
        const V* src = hs == 0 ? x : dst;
        const int t0 = (l0 ^ p) & 1;                 // first own level of parity p
        const int nh = n > t0 ? (n - t0 + 1) / 2 : 0;
        auto store = [&](int t, int i, V v) {
          if constexpr (sizeof(V) == 4) v += qv[t * m + i];
          dst[(t + 1) * m + i] = v;
          if (t == 0 && ha.left) push((last ? ha.zl : ha.xl) + i * (int)sizeof(V), ha.bl, v);
          if (t == n - 1 && ha.right) push((last ? ha.zr : ha.xr) + i * (int)sizeof(V), ha.br, v);
        };
        for_rows<V>(
            c, m, nh,
            [&](int u, int i, int j0, int S) {
              const int t = t0 + 2 * u;
              if (t == 0) halo_wait(ha, 0, kk, hs);
              if (t == n - 1) halo_wait(ha, 1, kk, hs);
              V sa = 1, sb = 1;
              if (sizeof(V) == 4 && h.sc) {
                sa = (V)h.sc[2 * (l0 + t)];
                sb = (V)h.sc[2 * (l0 + t) + 1];
              }
              return dot2(A + t * ms, B + t * ms, src + t * m, src + (t + 2) * m, m, i, j0, S, sa,
                          sb);
            },
            [&](int u, int i, V v) {
              if (COUPLED)
                store(t0 + 2 * u, i, v);
              else
                g[(t0 + 2 * u) * m + i] = v;
            });
        if (!COUPLED) {
          __syncthreads();
          for_rows<V>(
              c, m, nh,
              [&](int u, int i, int j0, int S) {
                const int t = t0 + 2 * u;
                return dot1(Cp + t * mc, g + t * m, m, i, j0, S);
              },
              [&](int u, int i, V v) { store(t0 + 2 * u, i, v); });
        }
        __syncthreads();
        halo_next(ha, kk, hs, K);
      }
    }
  }
  // the last version of a halo that only the next sweep would have read
#pragma unroll
  for (int side = 0; side < 2; ++side)
    if (ha.rh[side] == 0) halo_wait(ha, side, K, 0);
}

// Sums of three values over every CTA of the cluster, in a fixed order, on
// every thread.  The values of a CTA are in the first `warps` warps (v is
// ignored elsewhere): FP64 adds cost 16 clocks of the SM's pipe a warp, so no
// other warp takes part.  sh: kThreads / 32 + 1 triples of shared memory, a
// different array for every call.  Contains one cluster barrier.
__device__ __forceinline__ void cluster_sum3(double (&v)[3], int warps, double (*sh)[3]) {
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  double* own = sh[kThreads / 32];
  if (w < warps) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int i = 0; i < 3; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
    if (lane == 0)
      for (int i = 0; i < 3; ++i) (warps == 1 ? own : sh[w])[i] = v[i];
  }
  if (warps > 1) {
    __syncthreads();
    if (threadIdx.x < 3) {
      double t = sh[0][threadIdx.x];
      for (int i = 1; i < warps; ++i) t += sh[i][threadIdx.x];
      own[threadIdx.x] = t;
    }
  }
  cl.sync();
  if (w == 0) {
    const double* p = cl.map_shared_rank(own, lane < C ? lane : 0);
#pragma unroll
    for (int i = 0; i < 3; ++i) v[i] = lane < C ? p[i] : 0.0;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1)
#pragma unroll
      for (int i = 0; i < 3; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
    if (lane == 0)
      for (int i = 0; i < 3; ++i) sh[0][i] = v[i];   // own stays as it is for the other CTAs
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 3; ++i) v[i] = sh[0][i];
}

}  // namespace res
}  // namespace mc
