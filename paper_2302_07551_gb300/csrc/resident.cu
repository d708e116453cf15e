// Chains that stay on chip (resident_dev.cuh).  FP64: all sweeps of a call, the
// sums, the residual and the normalisation in one launch.  Low precision: the
// correction sweeps of a refinement step.
#include <math.h>

#include <mutex>

#include "batch.cuh"
#include "resident_dev.cuh"

namespace mc {

namespace {

using namespace res;

template <typename V>
__device__ __forceinline__ void attach(ClusterLink<V>& ln, const ResidentWords&, int* status) {
  ln.status = status;
  ln.c = (int)cg::this_cluster().num_blocks();
}
template <typename V>
__device__ __forceinline__ void attach(GridLink<V>& ln, const ResidentWords& w, int* status) {
  ln.first = w.first;
  ln.last = w.last;
  ln.g = reinterpret_cast<GridState*>(w.state);
  ln.status = status;
}

// The end of a launch: every CTA of a cluster stays until the others have read
// its shared memory; one CTA of a grid counts the versions up.
template <typename V>
__device__ __forceinline__ void finish(const ClusterLink<V>&) {
  cg::this_cluster().sync();
}
template <typename V>
__device__ __forceinline__ void finish(const GridLink<V>& ln) {
  ln.done();
}

// K FP64 sweeps from x_in, then x_out = z_K / e^T z_K with the step error
// (with_step) and ||Q^T x_out||_1 from the splitting (with_resid, see
// fused.cu) into the header and stats_out.  A solve runs several such chunks in
// one launch, the iterate staying on chip: a launch, a copy and a wait of the
// host per chunk of 32 sweeps were a third of a small solve (64 levels of 8 to
// 1e-12: 3.8 -> 3.0 ms).
template <bool COUPLED, typename Link>
__global__ void __launch_bounds__(kThreads, 1) k_resident(ResidentArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double sh[2][kThreads / 32 + 1][3];
  __shared__ double rcp[2];
  __shared__ unsigned long long two[2];
  Link ln;
  attach(ln, a.words, &a.hdr->status);
  const int C = ln.ctas(), r = ln.rank();
  Chain<double, double, double> h{};
  h.A = a.A;
  h.B = a.B;
  h.C = a.C;
  h.as = h.cs = a.ms;
  h.in = a.x_in;
  h.L = (int)a.L;
  h.m = a.m;
  h.par0 = a.par0;
  const int L = h.L, m = h.m;
  const int l0 = range_begin(L, C, r), n = range_begin(L, C, r + 1) - l0;
  const Carve k = carve<double, double, double, COUPLED>((L + C - 1) / C, m);
  double* x = reinterpret_cast<double*>(smem + k.x);
  double* z = reinterpret_cast<double*>(smem + k.z);
  // sums by as few warps as keep about 8 entries a lane
  int warps = (n * m + 255) / 256;
  if (warps > kThreads / 32) warps = kThreads / 32;
  double step = nan(""), prev = nan("");
  for (int64_t chunk = 1;; ++chunk) {
    sweeps<double, double, double, COUPLED>(h, (int)a.K, smem, two, ln, chunk == 1);
    double v[3] = {0.0, 0.0, 0.0};   // e^T z_K, e^T z_{K-1}, ||Q^T z_K||_1
    for (int e = threadIdx.x; e < n * m && threadIdx.x < 32 * warps; e += 32 * warps) {
      v[0] += z[m + e];
      if (a.K > 1) v[1] += x[m + e];
    }
    if (a.with_resid) {
      // N (x - z) on the diagonal-only rows: T_lo d_{l-1} + T_up d_{l+1}, d = z - x
      const int t0 = (l0 ^ a.par0) & 1, nh = n > t0 ? (n - t0 + 1) / 2 : 0;
      const Cover c = cover(m, (n + 1) / 2);
      double* rs = reinterpret_cast<double*>(smem + k.g);   // |r| per row
      for_rows<double>(
          c, m, nh, reinterpret_cast<double*>(smem + k.p),
          [&](int u, int i, int j0, int S) {
            const int t = t0 + 2 * u;
            const int64_t l = l0 + t;
            const double* A = a.TLO + (size_t)l * a.ms;   // once a chunk: from L2
            const double* B = a.TUP + (size_t)l * a.ms;
            // d at a halo beyond the chain is 0 - 0 and its block zero
            double s0 = 0.0;
#pragma unroll 4
            for (int j = j0; j < m; j += S) {
              s0 = fma(A[j * m + i], z[t * m + j] - x[t * m + j], s0);
              s0 = fma(B[j * m + i], z[(t + 2) * m + j] - x[(t + 2) * m + j], s0);
            }
            return s0;
          },
          [&](int u, int i, double s) { rs[u * m + i] = fabs(s); });
      __syncthreads();
      for (int e = threadIdx.x; e < nh * m && threadIdx.x < 32 * warps; e += 32 * warps)
        v[2] += rs[e];
    }
    all_sum3(v, warps, sh[0], ln, a.part);
    const double s = v[0], so = a.K > 1 ? v[1] : 1.0, res = v[2];
    // divisions are many FP64 instructions: one thread each, of different warps
    if (threadIdx.x == 0) rcp[0] = 1.0 / s;
    if (threadIdx.x == 32) rcp[1] = a.K > 1 ? 1.0 / so : 1.0;
    __syncthreads();
    const double inv = rcp[0], pinv = rcp[1];
    double w[3] = {0.0, 0.0, 0.0};
    if (a.with_step) {
      for (int e = threadIdx.x; e < n * m && threadIdx.x < 32 * warps; e += 32 * warps)
        w[0] += fabs(z[m + e] * inv - x[m + e] * pinv);
      all_sum3(w, warps, sh[1], ln, a.part + 3 * C);   // no CTA reads sh[0] of another after it
      prev = step;
      step = w[0];
    }
    const double resid = a.with_resid ? res * inv : nan("");
    const bool ok = s > 0.0 && isfinite(s);
    // the same decision in every CTA
    if (!ok || chunk >= a.chunks || (a.tol > 0.0 && resid <= a.tol) ||
        (a.eps > 0.0 && step <= a.eps)) {
      for (int e = threadIdx.x; e < n * m; e += kThreads)
        a.x_out[(int64_t)l0 * m + e] = z[m + e] * inv;
      if (r == 0 && threadIdx.x == 0) {
        if (!ok) latch(a.hdr, MC_ERR_BREAKDOWN);
        const double st[3] = {a.K > 1 ? s / so : s, w[0], resid};
        for (int i = 0; i < 3; ++i) {
          a.hdr->stats[i] = st[i];
          if (a.stats_out) a.stats_out[i] = st[i];
        }
        a.hdr->prev_step = prev;
        a.hdr->chunks = chunk;
      }
      break;
    }
    for (int e = threadIdx.x; e < (n + 2) * m; e += kThreads) x[e] = z[e] * inv;
    // (the next run's barrier comes before any CTA writes another's halo)
  }
  finish(ln);
}

// The K correction sweeps of a refinement step from the zero vector.
template <typename S, bool COUPLED, template <typename> class LinkT>
__global__ void __launch_bounds__(kThreads, 1) k_resident_lp(ResidentLpArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ unsigned long long two[2];
  LinkT<float> ln;
  attach(ln, a.words, &a.hdr->status);
  Chain<S, float, float> h{};
  h.A = reinterpret_cast<const S*>(a.A);
  h.B = reinterpret_cast<const S*>(a.B);
  h.C = a.C;
  h.as = a.abs_;
  h.cs = a.cbs;
  h.sc = a.sc;
  h.q = a.q;
  h.L = (int)a.L;
  h.m = a.m;
  h.par0 = a.par0;
  sweeps<S, float, float, COUPLED>(h, (int)a.K, smem, two, ln);
  const int l0 = ln.s.l0, n = ln.s.n;
  for (int e = threadIdx.x; e < n * h.m; e += kThreads)
    a.d[(int64_t)l0 * h.m + e] = ln.s.x[h.m + e];
  finish(ln);
}

// CTAs of a cluster of `most` that share L levels, at least two each.
__host__ __device__ inline int cluster_ctas(int64_t L, int most) {
  int C = most;
  while (C > 1 && L < 2 * C) C /= 2;
  return C;
}

// Dynamic shared memory of this launch: a request whose share does not fit it (none
// does not: its group follows from its size) is reported and left out.
__device__ __forceinline__ unsigned dyn_smem() {
  unsigned v;
  asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(v));
  return v;
}

// The resident requests of a group of a batch, one cluster each in turn; the CTAs of
// a short chain's cluster that have no levels only take part in its barriers.
// GROUP: the first group of this kernel.
template <typename S, bool COUPLED, int GROUP>
__global__ void __launch_bounds__(kThreads, group_share(GROUP))
    k_b_resident(const BTable* __restrict__ t, int group, int K, BOut* out) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ unsigned long long two[2];
  cg::cluster_group cl = cg::this_cluster();
  const int most = (int)cl.num_blocks(), cid = (int)blockIdx.x / most;
  const int clusters = t->res_clusters[group];
  if (cid >= clusters) return;
  const int i1 = t->res_end[group];
  for (int i = (group > 0 ? t->res_end[group - 1] : 0) + cid; i < i1; i += clusters) {
    const int r = t->res[i];
    const BReq& Q = t->r[r];
    ClusterLink<float> ln;
    ln.status = &out[r].status;
    ln.c = cluster_ctas(Q.L, most);
    if (Q.smem > (int)dyn_smem()) {
      atomicCAS(ln.status, 0, (int)MC_ERR_CUDA);
      continue;   // the whole cluster
    }
    if ((int)cl.block_rank() < ln.c) {
      Chain<S, float, float> h{};
      h.A = reinterpret_cast<const S*>(Q.lA);
      h.B = reinterpret_cast<const S*>(Q.lB);
      h.C = Q.lC;
      h.as = Q.lp_bs;
      h.cs = Q.lp_cbs;
      h.sc = Q.sc;
      h.q = Q.q;
      h.L = (int)Q.L;
      h.m = Q.m;
      h.par0 = Q.p1;
      sweeps<S, float, float, COUPLED, group_wide(GROUP)>(h, K, smem, two, ln);
      const int l0 = ln.s.l0, n = ln.s.n;
      for (int e = threadIdx.x; e < n * h.m; e += kThreads)
        Q.d[(int64_t)l0 * h.m + e] = ln.s.x[h.m + e];
    } else {
      ln.ready();
    }
    cl.sync();   // shared memory and barriers are used again
    if ((int)cl.block_rank() < ln.c && threadIdx.x == 0) {
      bar_free(ln.bar[0]);
      bar_free(ln.bar[1]);
    }
  }
}

// FP64: also the level sums of the last two sweeps, for the batch's reductions.
template <bool COUPLED>
__global__ void __launch_bounds__(kThreads, 1)
    k_b_resident64(const BTable* __restrict__ t, int group, int K, BOut* out) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ unsigned long long two[2];
  cg::cluster_group cl = cg::this_cluster();
  const int most = (int)cl.num_blocks(), cid = (int)blockIdx.x / most;
  const int clusters = t->res_clusters[group];
  if (cid >= clusters) return;
  const int i1 = t->res_end[group];
  for (int i = (group > 0 ? t->res_end[group - 1] : 0) + cid; i < i1; i += clusters) {
    const int r = t->res[i];
    const BReq& Q = t->r[r];
    ClusterLink<double> ln;
    ln.status = &out[r].status;
    ln.c = cluster_ctas(Q.L, most);
    if (Q.smem > (int)dyn_smem()) {
      atomicCAS(ln.status, 0, (int)MC_ERR_CUDA);
      continue;   // the whole cluster
    }
    if ((int)cl.block_rank() < ln.c) {
      Chain<double, double, double> h{};
      h.A = Q.A;
      h.B = Q.B;
      h.C = Q.C;
      h.as = h.cs = Q.ms;
      h.in = Q.x;
      h.L = (int)Q.L;
      h.m = Q.m;
      h.par0 = Q.p1;
      sweeps<double, double, double, COUPLED>(h, K, smem, two, ln);
      const int l0 = ln.s.l0, n = ln.s.n, m = h.m;
      for (int e = threadIdx.x; e < n * m; e += kThreads) {
        Q.z[(int64_t)l0 * m + e] = ln.s.z[m + e];
        if (K > 1) Q.xb[(int64_t)l0 * m + e] = ln.s.x[m + e];
      }
      for (int q = threadIdx.x; q < 2 * n; q += kThreads) {   // in row order
        const int lev = q >> 1, prev = q & 1;
        const double* v = (prev ? ln.s.x : ln.s.z) + (lev + 1) * m;
        double sum = 0.0;
        for (int j = 0; j < m; ++j) sum += v[j];
        if (!prev || K > 1) Q.lsum2[((K - 1 - prev) & 1) * Q.L + l0 + lev] = sum;
      }
    } else {
      ln.ready();
    }
    cl.sync();   // shared memory and barriers are used again
    if ((int)cl.block_rank() < ln.c && threadIdx.x == 0) {
      bar_free(ln.bar[0]);
      bar_free(ln.bar[1]);
    }
  }
}

constexpr size_t kMaxDyn = 227 * 1024 - 1024;   // opt-in limit less the static arrays

// Kernels by storage type (FP64, FP32, BF16), apply mode and link.
using Kernel64 = void (*)(ResidentArgs);
using KernelLp = void (*)(ResidentLpArgs);
using KernelBatch = void (*)(const BTable*, int, int, BOut*);
template <int GROUP>
KernelBatch kernel_batch_lp(int lp, int coupled) {
  if (lp == 1) return coupled ? k_b_resident<float, true, GROUP> : k_b_resident<float, false, GROUP>;
  return coupled ? k_b_resident<unsigned short, true, GROUP>
                 : k_b_resident<unsigned short, false, GROUP>;
}
KernelBatch kernel_batch(int lp, int coupled, int group) {
  if (lp == 0) return coupled ? k_b_resident64<true> : k_b_resident64<false>;
  return group < 2    ? kernel_batch_lp<0>(lp, coupled)
         : group == 2 ? kernel_batch_lp<2>(lp, coupled)
         : group == 3 ? kernel_batch_lp<3>(lp, coupled)
                      : kernel_batch_lp<4>(lp, coupled);
}
// Dynamic shared memory of a group's CTAs: an SM's 228 KB by the CTAs that share it,
// less 1 KB each and the static arrays.
size_t group_smem(int group) {
  const int n = group_share(group);
  return n == 1 ? kMaxDyn : (size_t)(228 / n - 2) * 1024;
}
Kernel64 kernel64(int coupled, bool grid) {
  if (grid)
    return coupled ? k_resident<true, GridLink<double>> : k_resident<false, GridLink<double>>;
  return coupled ? k_resident<true, ClusterLink<double>> : k_resident<false, ClusterLink<double>>;
}
template <typename S>
KernelLp kernel_lp_of(int coupled, bool grid) {
  if (grid) return coupled ? k_resident_lp<S, true, GridLink> : k_resident_lp<S, false, GridLink>;
  return coupled ? k_resident_lp<S, true, ClusterLink> : k_resident_lp<S, false, ClusterLink>;
}
KernelLp kernel_lp(int lp, int coupled, bool grid) {
  return lp == 1 ? kernel_lp_of<float>(coupled, grid) : kernel_lp_of<unsigned short>(coupled, grid);
}

size_t smem_bytes(const Layout& y, int coupled, int C) {
  const int n = (int)((y.L + C - 1) / C), m = y.m;
  if (y.lp == 0)
    return coupled ? carve<double, double, double, true>(n, m).total
                   : carve<double, double, double, false>(n, m).total;
  if (y.lp == 1)
    return coupled ? carve<float, float, float, true>(n, m).total
                   : carve<float, float, float, false>(n, m).total;
  return coupled ? carve<unsigned short, float, float, true>(n, m).total
                 : carve<unsigned short, float, float, false>(n, m).total;
}

void config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute& at, bool grid, int C, size_t smem,
            cudaStream_t s) {
  cfg.gridDim = dim3(C);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  if (grid) {
    at.id = cudaLaunchAttributeCooperative;
    at.val.cooperative = 1;
  } else {
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = C;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
  }
  cfg.attrs = &at;
  cfg.numAttrs = 1;
}

// Whether a cluster of C CTAs with all of an SM's shared memory can run.
bool cluster_runs(const void* kernel, int C) {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  config(cfg, at, false, C, kMaxDyn, 0);
  int n = 0;
  return cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess && n > 0;
}

bool opt_in(const void* kernel, bool cluster) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)kMaxDyn) == cudaSuccess &&
         (!cluster || cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed,
                                           1) == cudaSuccess);
}

// What the current device allows, found once per device: the largest cluster
// (16, the non-portable opt-in, 8 or 0) and the SMs of a cooperative launch with
// one CTA each (0: none).
struct Limits {
  bool known;
  int cluster, grid;
};
Limits limits() {
  constexpr int kDevices = 64;
  static std::mutex mu;
  static Limits all[kDevices];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevices) return Limits{};
  std::lock_guard<std::mutex> lk(mu);
  Limits& l = all[dev];
  if (!l.known) {
    bool ok = true;
    for (int c = 0; c < 2; ++c) {
      ok = ok && opt_in((const void*)kernel64(c, false), true) &&
           opt_in((const void*)kernel64(c, true), false) &&
           opt_in((const void*)kernel_batch(0, c, 1), true);
      for (int lp = 1; lp <= 2; ++lp)
        ok = ok && opt_in((const void*)kernel_lp(lp, c, false), true) &&
             opt_in((const void*)kernel_lp(lp, c, true), false) &&
             opt_in((const void*)kernel_batch(lp, c, 0), true) &&
             opt_in((const void*)kernel_batch(lp, c, 2), true) &&
             opt_in((const void*)kernel_batch(lp, c, 3), true) &&
             opt_in((const void*)kernel_batch(lp, c, 4), true);
    }
    if (ok) {
      for (int C = 16; C >= 8 && !l.cluster; C /= 2) {
        bool runs = true;
        for (int c = 0; c < 2; ++c) {
          runs = runs && cluster_runs((const void*)kernel64(c, false), C) &&
                 cluster_runs((const void*)kernel_batch(0, c, 1), C);
          for (int lp = 1; lp <= 2; ++lp)
            runs = runs && cluster_runs((const void*)kernel_lp(lp, c, false), C) &&
                   cluster_runs((const void*)kernel_batch(lp, c, 0), C) &&
                   cluster_runs((const void*)kernel_batch(lp, c, 2), C) &&
                   cluster_runs((const void*)kernel_batch(lp, c, 3), C) &&
                   cluster_runs((const void*)kernel_batch(lp, c, 4), C);
        }
        if (runs) l.cluster = C;
      }
      int sms = 0, coop = 0;
      if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
          cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess && coop)
        l.grid = sms;
    }
    cudaGetLastError();
    l.known = true;
  }
  return l;
}

}  // namespace

// Every CTA owns at least two levels (one of each parity).  A cluster (short
// hops) while its 16 SMs keep up: FP64 up to 96 K multiply-adds a sweep (3000
// clocks of the 32 FP64 lanes a clock), low precision up to 64 KB of shared
// memory a CTA (500 clocks of its bandwidth); else all SMs.
int resident_ctas(const Layout& y, int coupled, int* grid) {
  *grid = 0;
  if (y.L > (1 << 20)) return 0;
  const Limits lim = limits();
  const int C = cluster_ctas(y.L, lim.cluster);
  const double entries = (double)y.L * y.m * y.m * (coupled ? 2 : 3);
  const size_t most = y.lp ? 64 * 1024 : kMaxDyn;
  // low precision, m > 32: the team kernel (lpteam_dev.cuh) keeps more warps on a
  // level and is faster where it applies (500 levels of 64, FP32 inverse, 3.4 us a
  // sweep against 4.6)
  if (y.lp && y.m > 32 && (y.lp == 1 || y.m % 8 == 0)) return 0;
  if (C > 0 && smem_bytes(y, coupled, C) <= most && (y.lp || entries <= 96e3)) return C;
  int G = lim.grid;
  if (G > y.L / 2) G = (int)(y.L / 2);
  if (G > 0 && smem_bytes(y, coupled, G) <= kMaxDyn) {
    *grid = 1;
    return G;
  }
  return 0;
}

cudaError_t launch_resident(const ResidentArgs& a, const Layout& y, int coupled, int ctas,
                            int grid, cudaStream_t s) {
  if (y.lp != 0) return cudaErrorInvalidValue;   // ctas and smem_bytes follow the storage type
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  config(cfg, at, grid != 0, ctas, smem_bytes(y, coupled, ctas), s);
  return cudaLaunchKernelEx(&cfg, kernel64(coupled, grid != 0), a);
}

cudaError_t launch_resident_lp(const ResidentLpArgs& a, const Layout& y, int coupled, int ctas,
                               int grid, cudaStream_t s) {
  if (y.lp == 0) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  config(cfg, at, grid != 0, ctas, smem_bytes(y, coupled, ctas), s);
  return cudaLaunchKernelEx(&cfg, kernel_lp(y.lp, coupled, grid != 0), a);
}

int resident_cluster() { return limits().cluster; }

int resident_batch_group(const Layout& y, int coupled) {
  const int C = cluster_ctas(y.L, limits().cluster);
  if (C == 0 || y.m > 32 || y.L > (1 << 20)) return -1;
  const size_t need = smem_bytes(y, coupled, C);
  if (need > kMaxDyn) return -1;
  if (y.lp == 0) return 1;
  int g = y.m > 16 ? 2 : 0;
  while (need > group_smem(g)) ++g;
  return g;
}

int resident_batch_smem(const Layout& y, int coupled) {
  return (int)smem_bytes(y, coupled, cluster_ctas(y.L, limits().cluster));
}

void resident_order(const Layout& y, int16_t* c, int16_t* s) {
  *c = (int16_t)cluster_ctas(y.L, limits().cluster);
  const int n_half = (int)(((y.L + *c - 1) / *c + 1) / 2);
  const Cover v = cover(y.m, n_half);
  *s = (int16_t)(v.S > 1 ? v.S : is_tiny(y.m, n_half, v) ? 1 : 0);
}

cudaError_t launch_resident_batch(const BTable* t, int lp, int coupled, int group, int K, BOut* out,
                                  cudaStream_t s) {
  const int C = limits().cluster;
  if (C == 0) return cudaSuccess;   // no request has this path
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  config(cfg, at, false, C, group_smem(group), s);
  cfg.gridDim = dim3(C * kResidentSlots * group_share(group));
  return cudaLaunchKernelEx(&cfg, kernel_batch(lp, coupled, group), t, group, K, out);
}

}  // namespace mc
