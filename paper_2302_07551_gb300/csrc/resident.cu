// Small chains: all sweeps of a call, the sums, the residual and the
// normalisation in one launch of one thread-block cluster
// (resident_dev.cuh).
#include <math.h>

#include <mutex>

#include "resident_dev.cuh"

namespace mc {

namespace {

using namespace res;

// K FP64 sweeps from x_in, then x_out = z_K / e^T z_K with the step error
// (with_step) and ||Q^T x_out||_1 from the splitting (with_resid, see
// fused.cu) into the header and stats_out.
template <bool COUPLED>
__global__ void __launch_bounds__(kThreads) k_resident(ResidentArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double sh[2][kThreads / 32 + 1][3];
  __shared__ double rcp[2];
  __shared__ unsigned long long bars[2];
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), r = (int)cl.block_rank();
  Chain<double, double, double> h{};
  h.A = a.A;
  h.B = a.B;
  h.C = a.C;
  h.as = h.cs = a.ms;
  h.in = a.x_in;
  h.L = (int)a.L;
  h.m = a.m;
  h.par0 = a.par0;
  sweeps<double, double, double, COUPLED>(h, (int)a.K, smem, bars, &a.hdr->status);
  const int L = h.L, m = h.m;
  const int l0 = range_begin(L, C, r), n = range_begin(L, C, r + 1) - l0;
  const Carve k = carve<double, double, double, COUPLED>((L + C - 1) / C, m);
  const double* x = reinterpret_cast<double*>(smem + k.x);
  const double* z = reinterpret_cast<double*>(smem + k.z);
  double v[3] = {0.0, 0.0, 0.0};   // e^T z_K, e^T z_{K-1}, ||Q^T z_K||_1
  // sums by as few warps as keep about 8 entries a lane
  int warps = (n * m + 255) / 256;
  if (warps > kThreads / 32) warps = kThreads / 32;
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
        c, m, nh,
        [&](int u, int i, int j0, int S) {
          const int t = t0 + 2 * u;
          const int64_t l = l0 + t;
          const double* A = a.TLO + (size_t)l * a.ms;   // once a launch: from L2
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
  cluster_sum3(v, warps, sh[0]);
  const double s = v[0], so = a.K > 1 ? v[1] : 1.0, res = v[2];
  if (threadIdx.x == 0) {   // divisions are many FP64 instructions: one thread
    rcp[0] = 1.0 / s;
    rcp[1] = a.K > 1 ? 1.0 / so : 1.0;
  }
  __syncthreads();
  const double inv = rcp[0], pinv = rcp[1];
  double w[3] = {0.0, 0.0, 0.0};
  for (int e = threadIdx.x; e < n * m && threadIdx.x < 32 * warps; e += 32 * warps) {
    const double p = z[m + e] * inv;
    if (a.with_step) w[0] += fabs(p - x[m + e] * pinv);
    a.x_out[(int64_t)l0 * m + e] = p;
  }
  cluster_sum3(w, warps, sh[1]);   // after its barrier no CTA reads sh[0] of another
  if (r == 0 && threadIdx.x == 0) {
    if (!((s > 0.0) && isfinite(s))) latch(a.hdr, MC_ERR_BREAKDOWN);
    const double st[3] = {a.K > 1 ? s / so : s, w[0], a.with_resid ? res * inv : nan("")};
    for (int i = 0; i < 3; ++i) {
      a.hdr->stats[i] = st[i];
      if (a.stats_out) a.stats_out[i] = st[i];
    }
  }
  cl.sync();   // every CTA stays until the others have read its sums
}

constexpr size_t kMaxDyn = 227 * 1024 - 1024;   // opt-in limit less the static arrays

// Whether a cluster of C CTAs with all of an SM's shared memory can run.
template <typename K>
bool cluster_runs(K kernel, int C) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(C);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kMaxDyn;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = C;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  int n = 0;
  return cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess && n > 0;
}

template <typename K>
bool opt_in(K kernel) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)kMaxDyn) == cudaSuccess &&
         cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
             cudaSuccess;
}

// Largest cluster of the current device: 16 (the non-portable opt-in), 8 or
// none; found once per device.
int cluster_limit() {
  constexpr int kDevices = 64;
  static std::mutex mu;
  static int limit[kDevices];   // 0: not asked yet, -1: none
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevices) return 0;
  std::lock_guard<std::mutex> lk(mu);
  if (limit[dev] == 0) {
    limit[dev] = -1;
    if (opt_in(k_resident<true>) && opt_in(k_resident<false>))
      for (int C = 16; C >= 8; C /= 2)
        if (cluster_runs(k_resident<true>, C) && cluster_runs(k_resident<false>, C)) {
          limit[dev] = C;
          break;
        }
    cudaGetLastError();
  }
  return limit[dev] > 0 ? limit[dev] : 0;
}

template <bool C>
cudaError_t launch(const ResidentArgs& a, int cluster, cudaStream_t s) {
  const int n = (int)((a.L + cluster - 1) / cluster);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(cluster);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = carve<double, double, double, C>(n, a.m).total;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = cluster;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_resident<C>, a);
}

}  // namespace

// The largest cluster that leaves every CTA two levels (one of each parity), if
// the chain fits its shared memory.
int resident_cluster(const Layout& y, int coupled) {
  if (y.L > (1 << 20)) return 0;
  int C = cluster_limit();
  while (C > 1 && y.L < 2 * C) C /= 2;
  if (C < 1) return 0;
  const int n = (int)((y.L + C - 1) / C);
  const size_t bytes = coupled ? carve<double, double, double, true>(n, y.m).total
                               : carve<double, double, double, false>(n, y.m).total;
  return bytes <= kMaxDyn ? C : 0;
}

cudaError_t launch_resident(const ResidentArgs& a, int coupled, int cluster, cudaStream_t s) {
  return coupled ? launch<true>(a, cluster, s) : launch<false>(a, cluster, s);
}

}  // namespace mc
