// Staircase sweeps of a chain that stays on chip: every CTA of the launch owns a
// contiguous range of levels, loads their operators once, and exchanges the
// two boundary levels of its range with its neighbours every half-sweep.
//
// A small chain's sweep through global memory (k_sweeps, k_sweeps_lp) is a
// serial chain of L2 round trips: the wait for the neighbours' counters, their
// acquire, the vectors, each operator block, the fence and the release, 5.3 us
// per half-sweep whatever the arithmetic.  On chip, FP64: 64 levels of 8 (cluster)
// 10.7 -> 1.25 us a sweep (coupled 7.9 -> 0.91), 1500 levels of 8 (all SMs) 12.6 ->
// 2.2, 130 levels of 32 17 -> 5.6; 1024 levels of 16, BF16 coupled, 8.6 -> 1.7.
// What is left of a small FP64 sweep is the pipe's 64 clocks per instruction and
// warp, 11 of them in a row per half-sweep, and the exchange.
//
// Two links between the CTAs:
//   ClusterLink (chains that fit 16 SMs and keep them fast enough): one
//     thread-block cluster; boundary levels are pushed into the neighbour's
//     shared memory.  The hardware co-schedules a cluster.
//   GridLink (chains that fit all SMs): a cooperative launch; boundary levels
//     travel through L2 as words that carry their version, polled by the reader.
//     A hop takes about 0.42 us instead of 0.17.
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
  size_t a, b, c, x, z, g, p, s, total;
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
  k.p = o;   // partial sums (for_rows; low precision: four rows a thread)
  o += kThreads * (sizeof(V) == 8 ? 8 : 16);
  k.s = o;   // low precision: block scales
  if (sizeof(V) == 4) o += up(2 * (size_t)n * sizeof(float));
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
__host__ __device__ inline Cover cover(int m, int n_half) {
  Cover c{1, 1, 1};
  if (m > 16) return c;
  while (c.mp < m) c.mp *= 2;
  while (c.mp * c.S < 32 && c.S < m && n_half * c.mp * c.S * 2 <= kThreads) c.S *= 2;
  c.gs = c.mp * c.S;
  return c;
}

// Whether the operators fit the threads' registers (sweeps_tiny).
__host__ __device__ inline bool is_tiny(int m, int n_half, const Cover& c) {
  return m <= 16 && n_half * c.gs <= kThreads && (m + c.S - 1) / c.S <= 8;
}

// Column groups of flattened rows of a half-sweep (for_rows): with fewer than 32 rows
// per sub-partition (each has its own FP64 pipe) the columns are split over warps as
// well, and the parts of a row added in order.
__host__ __device__ inline int flat_split(int rows) {
  const int chunks = (rows + 31) / 32;
  return chunks * 2 <= 4 ? 4 / chunks : 1;
}

// sum_j A(i, j) p_j + B(i, j) q_j over this thread's columns, in one chain: a
// warp's FP64 instructions issue 64 clocks apart anyway.
__device__ __forceinline__ double dot2(const double* A, const double* B, const double* p,
                                       const double* q, int m, int i, int j0, int S) {
  double a = 0.0;
  const double *pa = A + j0 * m + i, *pb = B + j0 * m + i;
#pragma unroll 4
  for (int j = j0; j < m; j += S, pa += S * m, pb += S * m) {
    a = fma(*pa, p[j], a);
    a = fma(*pb, q[j], a);
  }
  return a;
}

__device__ __forceinline__ double dot1(const double* A, const double* p, int m, int i, int j0,
                                       int S) {
  double a = 0.0;
  const double* pa = A + j0 * m + i;
#pragma unroll 4
  for (int j = j0; j < m; j += S, pa += S * m) a = fma(*pa, p[j], a);
  return a;
}

// value(u, i, j0, S) per (level u of the half-sweep's n_half, row i): the part of
// the row's sum over columns j0, j0 + S, ...; then store(u, i, sum).  Warps
// without rows issue nothing.  part: kThreads values of shared memory.
template <typename V, typename F, typename G>
__device__ __forceinline__ void for_rows(const Cover& c, int m, int n_half, V* part, F value,
                                         G store) {
  if (c.S == 1) {
    const int rows = n_half * m, chunks = (rows + 31) / 32;
    const int S = flat_split(rows);
    if (S == 1) {
      for (int t = threadIdx.x; t < rows; t += kThreads) {
        const int u = t / m, i = t - u * m;
        store(u, i, value(u, i, 0, 1));
      }
      return;
    }
    const int w = threadIdx.x >> 5, s = w / chunks;
    const int row = (w - s * chunks) * 32 + (threadIdx.x & 31);
    if (s < S && row < rows) part[s * chunks * 32 + row] = value(row / m, row % m, s, S);
    __syncthreads();
    for (int t = threadIdx.x; t < rows; t += kThreads) {
      V v = part[t];
      for (int q = 1; q < S; ++q) v += part[q * chunks * 32 + t];
      store(t / m, t % m, v);
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
// A halo gets one version per sweep: the neighbour writes its boundary level
// once a sweep.  It can only write the next one after it has received this
// CTA's own boundary level, computed after the read, so no version is
// overwritten before it was read.
//
// Half-sweep hs of sweep kk reads a halo if rh = hs (the half-sweep of the
// boundary level's parity); kk + hs versions must have arrived by then.
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
__device__ __forceinline__ void bar_free(uint32_t bar) {
  asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void bar_expect(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}

// Bounded spinning: true when a wait should be given up, after 2 s of the
// global timer (then MC_ERR_TIMEOUT is latched) or once that error is latched,
// so that a launch always ends.
struct Spin {
  unsigned long long t0 = 0;
  int it = 0;
  __device__ __forceinline__ bool give_up(int* status) {
    if ((it++ & 255) != 0) return false;
    if (t0 == 0) {
      t0 = dev::global_ns();
      return false;
    }
    if (*reinterpret_cast<volatile int*>(status) == (int)MC_ERR_TIMEOUT) return true;
    if (dev::global_ns() - t0 <= 2000000000ull) return false;
    atomicCAS(status, 0, (int)MC_ERR_TIMEOUT);
    return true;
  }
};

// Wait for the completion of the mbarrier phase of this parity.
__device__ __forceinline__ void bar_wait(uint32_t bar, uint32_t parity, int* status) {
  Spin sp;
  while (true) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok || sp.give_up(status)) return;
  }
}

// Where a CTA's vectors are and which neighbours it has.
template <typename V>
struct Side {
  V *x, *z;
  int l0, n, m, par0, K;
  bool left, right;
  __device__ __forceinline__ int rh(int side) const {
    const int l = side == 0 ? l0 : l0 + n - 1;
    return (l & 1) == par0 ? 0 : 1;
  }
};

// Neighbours in the same cluster.  Every pushed version completes one phase of
// the receiver's mbarrier (m values of transaction bytes); about 350 clocks a
// half-sweep with the block barrier, against 660 for a cluster barrier behind a
// distributed store.
template <typename V>
struct ClusterLink {
  Side<V> s;
  uint32_t bar[2];                 // own barriers: left, right halo
  uint32_t xl, xr, zl, zr, bl, br; // the neighbours' halo slots and barriers
  int* status;
  int c;                           // CTAs that take part (the first c of the cluster)
  int used;                        // phases completed by earlier runs

  __device__ __forceinline__ int ctas() const { return c; }
  __device__ __forceinline__ int rank() const { return (int)cg::this_cluster().block_rank(); }
  // n_left: levels of the left neighbour.  bars: two mbarriers.
  __device__ __forceinline__ void open(const Side<V>& side, int n_left, unsigned long long* bars) {
    s = side;
    used = 0;
    const int r = rank();
    bar[0] = smem_addr(bars);
    bar[1] = smem_addr(bars + 1);
    if (s.left) {
      xl = peer_addr(smem_addr(s.x + (n_left + 1) * s.m), r - 1);
      zl = peer_addr(smem_addr(s.z + (n_left + 1) * s.m), r - 1);
      bl = peer_addr(bar[1], r - 1);
    }
    if (s.right) {
      xr = peer_addr(smem_addr(s.x), r + 1);
      zr = peer_addr(smem_addr(s.z), r + 1);
      br = peer_addr(bar[0], r + 1);
    }
    if (threadIdx.x == 0) {
      bar_init(bar[0]);
      bar_init(bar[1]);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    arm();
  }
  // the barriers expect the first version of a run of K sweeps
  __device__ __forceinline__ void arm() const {
    if (threadIdx.x == 0) {
      if (s.left) bar_expect(bar[0], (uint32_t)(s.m * sizeof(V)));
      if (s.right) bar_expect(bar[1], (uint32_t)(s.m * sizeof(V)));
    }
  }
  // another run after a finished one
  __device__ __forceinline__ void again() {
    used += s.K;
    arm();
  }
  // every CTA is ready for pushes
  __device__ __forceinline__ void ready() { cg::this_cluster().sync(); }
  __device__ __forceinline__ void fill(int, int) {}   // the halo arrives by itself
  __device__ __forceinline__ void wait(int side, int kk, int hs) const {
    const int need = kk + hs;
    if (need > 0 && (side == 0 ? s.left : s.right))
      bar_wait(bar[side], (uint32_t)(used + need - 1) & 1u, status);
  }
  // value i of boundary level t of sweep kk
  __device__ __forceinline__ void send(int t, int i, V v, int, bool last) const {
    if (t == 0 && s.left) push((last ? zl : xl) + i * (int)sizeof(V), bl, v);
    if (t == s.n - 1 && s.right) push((last ? zr : xr) + i * (int)sizeof(V), br, v);
  }
  // after the block barrier that ends a half-sweep (its readers have received
  // their versions): arm the barriers for the next ones, K versions in all
  __device__ __forceinline__ void next(int kk, int hs) const {
    if (threadIdx.x < 2) {
      const int side = threadIdx.x, need = kk + hs;
      if ((side == 0 ? s.left : s.right) && s.rh(side) == hs && need > 0 && need < s.K)
        bar_expect(bar[side], (uint32_t)(s.m * sizeof(V)));
    }
  }
  // the last version of a halo that only the next sweep would have read
  __device__ __forceinline__ void close() const {
#pragma unroll
    for (int side = 0; side < 2; ++side)
      if (s.rh(side) == 0) wait(side, s.K, 0);
  }
};

// Words (wave_dev.cuh) of a vector in global memory; a double takes two.
using dev::ld_word;
using dev::st_word;
__device__ __forceinline__ void put(unsigned long long* p, int i, float v, unsigned version) {
  st_word(p + i, __float_as_uint(v), version);
}
__device__ __forceinline__ void put(unsigned long long* p, int i, double v, unsigned version) {
  st_word(p + 2 * i, (unsigned)__double2loint(v), version);
  st_word(p + 2 * i + 1, (unsigned)__double2hiint(v), version);
}
__device__ __forceinline__ void get(const unsigned long long* p, int i, unsigned version, float* v,
                                    int* status) {
  unsigned long long w;
  Spin sp;
  do {
    w = ld_word(p + i);
  } while ((unsigned)(w >> 32) != version && !sp.give_up(status));
  *v = __uint_as_float((unsigned)w);
}
__device__ __forceinline__ void get(const unsigned long long* p, int i, unsigned version, double* v,
                                    int* status) {
  unsigned long long a, b;
  Spin sp;
  do {
    a = ld_word(p + 2 * i);
    b = ld_word(p + 2 * i + 1);
  } while (((unsigned)(a >> 32) != version || (unsigned)(b >> 32) != version) &&
           !sp.give_up(status));
  *v = __hiloint2double((int)(unsigned)b, (int)(unsigned)a);
}

// Shared counters of a cooperative launch (zero before the first launch of a
// chain, left ready for the next one).
struct GridState {
  unsigned arrived, generation;    // grid barrier
  unsigned joined, version;        // launches: versions used so far
};

// Neighbours anywhere on the GPU.  first / last: the CTAs' boundary levels,
// one row of words per CTA.  Versions go on from launch to launch, so the words
// need no reset.
template <typename V>
struct GridLink {
  Side<V> s;
  unsigned long long *first, *last;
  GridState* g;
  unsigned base;
  int* status;
  static constexpr int W = sizeof(V) / 4;   // words per value

  __device__ __forceinline__ int ctas() const { return (int)gridDim.x; }
  __device__ __forceinline__ int rank() const { return (int)blockIdx.x; }
  __device__ __forceinline__ void open(const Side<V>& side, int, unsigned long long* sh) {
    s = side;
    if (threadIdx.x == 0) {
      *sh = *reinterpret_cast<volatile unsigned*>(&g->version);
      __threadfence();
      atomicAdd(&g->joined, 1u);   // this CTA has read the version
    }
    __syncthreads();
    base = (unsigned)*reinterpret_cast<volatile unsigned long long*>(sh);
  }
  __device__ __forceinline__ void again() { base += (unsigned)s.K; }
  __device__ __forceinline__ void ready() { __syncthreads(); }
  // the halos that half-sweep hs of sweep kk reads, into shared memory
  __device__ __forceinline__ void fill(int kk, int hs) {
    const int need = kk + hs;
    if (need == 0) return;
    V* dst = sizeof(V) == 8 && need == s.K ? s.z : s.x;   // version K: the last sweep's
    bool any = false;
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      if (!(side == 0 ? s.left : s.right) || s.rh(side) != hs) continue;
      any = true;
      const unsigned long long* src = side == 0
                                          ? last + (size_t)(rank() - 1) * s.m * W
                                          : first + (size_t)(rank() + 1) * s.m * W;
      V* h = dst + (side == 0 ? 0 : (s.n + 1) * s.m);
      // the two sides' words by different threads
      for (int i = ((int)threadIdx.x + side * (kThreads / 2)) % kThreads; i < s.m; i += kThreads)
        get(src, i, base + (unsigned)need, h + i, status);
    }
    if (any) __syncthreads();
  }
  __device__ __forceinline__ void wait(int, int, int) const {}
  __device__ __forceinline__ void send(int t, int i, V v, int kk, bool) const {
    const size_t o = (size_t)rank() * s.m * W;
    if (t == 0 && s.left) put(first + o, i, v, base + (unsigned)kk + 1u);
    if (t == s.n - 1 && s.right) put(last + o, i, v, base + (unsigned)kk + 1u);
  }
  __device__ __forceinline__ void next(int, int) const {}
  __device__ __forceinline__ void close() {
    if (sizeof(V) == 8) fill(s.K, 0);   // halos read in first half-sweeps: the last version
  }
  // Every CTA arrives before any leaves.
  __device__ __forceinline__ void barrier() const {
    __syncthreads();
    if (threadIdx.x == 0) {
      const unsigned gen = *reinterpret_cast<volatile unsigned*>(&g->generation);
      __threadfence();
      if (atomicAdd(&g->arrived, 1u) == gridDim.x - 1) {
        g->arrived = 0u;
        __threadfence();
        atomicAdd(&g->generation, 1u);
      } else {
        Spin sp;
        while (*reinterpret_cast<volatile unsigned*>(&g->generation) == gen &&
               !sp.give_up(status)) {
        }
      }
      __threadfence();
    }
    __syncthreads();
  }
  // One CTA, at the end: the versions of this launch are used up.
  __device__ __forceinline__ void done() const {
    if (rank() == 0 && threadIdx.x == 0) {
      Spin sp;
      while (*reinterpret_cast<volatile unsigned*>(&g->joined) != gridDim.x &&
             !sp.give_up(status)) {
      }
      g->joined = 0u;
      g->version = base + (unsigned)s.K;
    }
  }
};

// Chains whose half-sweep gives every thread at most one (level, row, column
// group): the operators' entries stay in registers, CPL columns a lane and
// operator for both parities; the inverse's input moves between the lanes of
// a level by shuffles.
template <typename T, typename TC, typename V, bool COUPLED, int CPL, typename Link>
__device__ __forceinline__ void sweeps_tiny(const Chain<T, TC, V>& h, int K, const Cover& c,
                                            Link& ln) {
  V *x = ln.s.x, *z = ln.s.z;
  const int L = h.L, m = h.m, l0 = ln.s.l0, n = ln.s.n;
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
      ln.fill(kk, hs);
      if (busy[hs]) {
        const int t = tt[hs];
        if (ok[hs] && t == 0) ln.wait(0, kk, hs);
        if (ok[hs] && t == n - 1) ln.wait(1, kk, hs);
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
          ln.send(t, i, v, kk, last);
        }
      }
      __syncthreads();
      ln.next(kk, hs);
    }
  }
}

// ---- low precision, more rows than threads' worth of registers ---------------
// A thread takes four rows of a level (m % 4 == 0: 16 or 8 bytes of a column) and
// every S-th column, S as large as the half-sweep leaves threads; the S partial
// sums of a row are added in order through shared memory.  Shared-memory reads
// bound the half-sweep: four rows share one read of the vector entry, and few
// columns a thread keep the serial chain short (2048 levels of 24, FP32 inverse:
// 3.7 us a sweep with one row a thread, 3.1 with four; 10.8 through global memory).
__device__ __forceinline__ float4 quad(const float* p) {
  return *reinterpret_cast<const float4*>(p);
}
__device__ __forceinline__ float4 quad(const unsigned short* p) {
  const uint2 t = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(t.x << 16), __uint_as_float(t.x & 0xffff0000u),
                     __uint_as_float(t.y << 16), __uint_as_float(t.y & 0xffff0000u));
}
__device__ __forceinline__ void fma4(float4& a, const float4& b, float s) {
  a.x = fmaf(b.x, s, a.x);
  a.y = fmaf(b.y, s, a.y);
  a.z = fmaf(b.z, s, a.z);
  a.w = fmaf(b.w, s, a.w);
}

// Thread (u, s, i): level u of the half-sweep, column group s, rows i .. i + 3, with
// i fastest and u slowest: a warp reads neighbouring columns of one level, which
// are contiguous (rows fastest over levels would meet the same banks in every
// level).
struct QuadMap {
  int quads, S;            // row quads of the half-sweep, column groups
  int u, s, i;             // this thread's part (u < 0: none)
  int ru, ri;              // and the row whose sum it takes (ru < 0: none)
};
__device__ __forceinline__ QuadMap quad_map(int m, int nh) {
  QuadMap q;
  const int per = m / 4, t = threadIdx.x;
  q.quads = nh * per;
  q.S = kThreads / q.quads;
  if (q.S < 1) q.S = 1;
  if (q.S > m) q.S = m;
  q.u = t / (per * q.S);
  q.s = (t - q.u * per * q.S) / per;
  q.i = 4 * (t % per);
  if (q.u >= nh) q.u = -1;
  q.ru = t / m;
  q.ri = t - q.ru * m;
  if (q.ru >= nh) q.ru = -1;
  return q;
}

// body(u, i, s, S) -> float4 per row quad and column group, then store(u, i, sum)
// per row.  part: 4 kThreads floats.
template <typename F, typename G>
__device__ __forceinline__ void for_quads(const QuadMap& q, int m, int nh, float* part, F body,
                                          G store) {
  if (q.S == 1) {
    for (int t = threadIdx.x; t < q.quads; t += kThreads) {
      const int u = t / (m / 4), i = 4 * (t - u * (m / 4));
      const float4 v = body(u, i, 0, 1);
      store(u, i, v.x);
      store(u, i + 1, v.y);
      store(u, i + 2, v.z);
      store(u, i + 3, v.w);
    }
    return;
  }
  if (q.u >= 0)
    *reinterpret_cast<float4*>(part + 4 * threadIdx.x) = body(q.u, q.i, q.s, q.S);
  __syncthreads();
  int u = q.ru, i = q.ri;
  for (int t = threadIdx.x; t < 4 * q.quads; t += kThreads) {
    if (t >= kThreads) {
      u = t / m;
      i = t - u * m;
    }
    const float* p = part + u * q.S * m + i;
    float v = p[0];
#pragma unroll 4
    for (int k = 1; k < q.S; ++k) v += p[k * m];
    store(u, i, v);
  }
}

template <typename T, typename TC, bool COUPLED, typename Link>
__device__ __forceinline__ void sweeps_quads(const T* A, const T* B, const TC* C, const float* sc,
                                             const float* qv, float* g, float* part, int ms,
                                             int mc, int K, Link& ln) {
  const int m = ln.s.m, n = ln.s.n, l0 = ln.s.l0;
  float* x = ln.s.x;
  QuadMap q[2];
  int t0[2], nh[2];
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int p = e == 0 ? ln.s.par0 : 1 - ln.s.par0;
    t0[e] = (l0 ^ p) & 1;
    nh[e] = (n - t0[e] + 1) / 2;
    q[e] = quad_map(m, nh[e]);
  }
  for (int kk = 0; kk < K; ++kk) {
#pragma unroll
    for (int hs = 0; hs < 2; ++hs) {
      auto store = [&](int u, int i, float v) {
        const int t = t0[hs] + 2 * u;
        v += qv[t * m + i];
        x[(t + 1) * m + i] = v;
        ln.send(t, i, v, kk, false);
      };
      ln.fill(kk, hs);
      for_quads(
          q[hs], m, nh[hs], part,
          [&](int u, int i, int s, int S) {
            const int t = t0[hs] + 2 * u;
            if (t == 0) ln.wait(0, kk, hs);
            if (t == n - 1) ln.wait(1, kk, hs);
            const T *pa = A + t * ms + i, *pb = B + t * ms + i;
            const float *lo = x + t * m, *up = lo + 2 * m;
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
#pragma unroll 4
            for (int j = s; j < m; j += S) {
              fma4(a, quad(pa + j * m), lo[j]);
              fma4(b, quad(pb + j * m), up[j]);
            }
            const float sa = sc[2 * t], sb = sc[2 * t + 1];
            return make_float4(fmaf(a.x, sa, b.x * sb), fmaf(a.y, sa, b.y * sb),
                               fmaf(a.z, sa, b.z * sb), fmaf(a.w, sa, b.w * sb));
          },
          [&](int u, int i, float v) {
            if (COUPLED)
              store(u, i, v);
            else
              g[(t0[hs] + 2 * u) * m + i] = v;
          });
      if (!COUPLED) {
        __syncthreads();
        for_quads(
            q[hs], m, nh[hs], part,
            [&](int u, int i, int s, int S) {
              const int t = t0[hs] + 2 * u;
              const TC* pc = C + t * mc + i;
              const float* v = g + t * m;
              float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
              for (int j = s; j < m; j += S) fma4(a, quad(pc + j * m), v[j]);
              return a;
            },
            store);
      }
      __syncthreads();
      ln.next(kk, hs);
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
// sh: two words of shared memory for the link.  first = false: another run from
// the iterate in x (halos included), with the operators as they are.  WIDE: m > 16.
template <typename T, typename TC, typename V, bool COUPLED, bool WIDE = false, typename Link>
__device__ __forceinline__ void sweeps(const Chain<T, TC, V>& h, int K, unsigned char* smem,
                                       unsigned long long* sh, Link& ln, bool first = true) {
  const int C = ln.ctas(), r = ln.rank();
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
  V* part = reinterpret_cast<V*>(smem + k.p);
  V* qv = g + (COUPLED ? 0 : (size_t)nmax * m);
  const int tid = threadIdx.x;
  const Cover c = cover(m, (nmax + 1) / 2);   // the same in every CTA
  const int cpl = (m + c.S - 1) / c.S;
  const bool tiny = !WIDE && m <= 16 && ((nmax + 1) / 2) * c.gs <= kThreads && cpl <= 8;   // is_tiny
  if (first) {
    ln.open(Side<V>{x, z, l0, n, m, h.par0, K, r > 0, r < C - 1},
            r > 0 ? l0 - range_begin(L, C, r - 1) : 0, sh);
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
  } else {
    ln.again();
  }
  float* sc = reinterpret_cast<float*>(smem + k.s);
  if (sizeof(V) == 4 && !tiny) {
    for (int e = tid; e < n * m; e += kThreads) qv[e] = (V)h.q[(int64_t)l0 * m + e];
    for (int e = tid; e < 2 * n; e += kThreads) sc[e] = h.sc[2 * l0 + e];
  }
  ln.ready();
  if (!WIDE && tiny) {
    if (cpl <= 1)
      sweeps_tiny<T, TC, V, COUPLED, 1>(h, K, c, ln);
    else if (cpl <= 2)
      sweeps_tiny<T, TC, V, COUPLED, 2>(h, K, c, ln);
    else if (cpl <= 4)
      sweeps_tiny<T, TC, V, COUPLED, 4>(h, K, c, ln);
    else
      sweeps_tiny<T, TC, V, COUPLED, 8>(h, K, c, ln);
  } else if constexpr (sizeof(V) == 4) {
    sweeps_quads<T, TC, COUPLED>(A, B, Cp, sc, qv, g, part, ms, mc, K, ln);
  } else {
    for (int kk = 0; kk < K; ++kk) {
      const bool last = kk == K - 1;
      V* dst = last ? z : x;
#pragma unroll 1
      for (int hs = 0; hs < 2; ++hs) {
        const int p = hs == 0 ? h.par0 : 1 - h.par0;
        const V* src = hs == 0 ? x : dst;
        const int t0 = (l0 ^ p) & 1;                 // first own level of parity p
        const int nh = n > t0 ? (n - t0 + 1) / 2 : 0;
        auto store = [&](int t, int i, V v) {
          dst[(t + 1) * m + i] = v;
          ln.send(t, i, v, kk, last);
        };
        ln.fill(kk, hs);
        for_rows<V>(
            c, m, nh, part,
            [&](int u, int i, int j0, int S) {
              const int t = t0 + 2 * u;
              if (t == 0) ln.wait(0, kk, hs);
              if (t == n - 1) ln.wait(1, kk, hs);
              return dot2(A + t * ms, B + t * ms, src + t * m, src + (t + 2) * m, m, i, j0, S);
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
              c, m, nh, part,
              [&](int u, int i, int j0, int S) {
                const int t = t0 + 2 * u;
                return dot1(Cp + t * mc, g + t * m, m, i, j0, S);
              },
              [&](int u, int i, V v) { store(t0 + 2 * u, i, v); });
        }
        __syncthreads();
        ln.next(kk, hs);
      }
    }
  }
  ln.close();
}

// Sums of three values over a CTA, in a fixed order, into own (shared).  The
// values are in the first `warps` warps (v is ignored elsewhere): FP64 adds cost
// 16 clocks of the SM's pipe a warp, so no other warp takes part.
__device__ __forceinline__ void block_sum3(double (&v)[3], int warps, double (*sh)[3],
                                           double* own) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
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
}

// The CTAs' sums added in rank order (a fixed tree), on every thread of every
// CTA.  sh: kThreads / 32 + 1 triples, another array for every call.
__device__ __forceinline__ void all_sum3(double (&v)[3], int warps, double (*sh)[3],
                                         const ClusterLink<double>& ln, double*) {
  cg::cluster_group cl = cg::this_cluster();
  const int C = ln.ctas(), lane = threadIdx.x & 31;
  double* own = sh[kThreads / 32];
  block_sum3(v, warps, sh, own);
  cl.sync();
  if (threadIdx.x < 32) {
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
// part: one triple per CTA in global memory, another array for every call.
__device__ __forceinline__ void all_sum3(double (&v)[3], int warps, double (*sh)[3],
                                         const GridLink<double>& ln, double* part) {
  const int C = ln.ctas(), lane = threadIdx.x & 31;
  double* own = sh[kThreads / 32];
  block_sum3(v, warps, sh, own);
  __syncthreads();
  if (threadIdx.x < 3) part[3 * ln.rank() + threadIdx.x] = own[threadIdx.x];
  ln.barrier();
  if (threadIdx.x < 32) {
#pragma unroll
    for (int i = 0; i < 3; ++i) v[i] = 0.0;
    for (int c = lane; c < C; c += 32)
#pragma unroll
      for (int i = 0; i < 3; ++i) v[i] += __ldcg(part + 3 * c + i);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int i = 0; i < 3; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
    if (lane == 0)
      for (int i = 0; i < 3; ++i) sh[0][i] = v[i];
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 3; ++i) v[i] = sh[0][i];
}

}  // namespace res
}  // namespace mc
