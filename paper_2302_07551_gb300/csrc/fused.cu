// Several staircase sweeps (Algorithm 2, repeated) in one persistent launch.
//
// Work units are (sweep k, half-sweep h, level l), claimed in that order from
// one queue counter by teams of warps (team_dev.cuh).  Half-sweep 1 of sweep k (the diagonal-only stair rows)
// reads its neighbours as left by half-sweep 2 of sweep k-1; half-sweep 2
// reads its neighbours as left by half-sweep 1 of sweep k.  So each unit
// depends on exactly two earlier units, the neighbour levels l-1 and l+1, and
// waits for them through per-level completion counters instead of a launch
// boundary: the grid streams through all K sweeps with one ramp-up and one
// tail, and the queue balances the load across warps and SMs.
//
// The vector is updated in place (W).  A unit overwrites level l only after
// both units that read the old value of level l (its neighbours' previous
// updates) have completed, which is exactly the condition it waits for.  The
// last sweep writes Z instead, so that W keeps z_{K-1} for the step error.
//
// Progress: a team handles its claimed units in increasing queue order and
// every unit depends only on units earlier in the queue, all claimed by
// running teams, so the earliest unfinished unit can always proceed.  Each
// wait is still bounded (FusedArgs::wait_ns of the GPU's global timer); on
// expiry the warp latches MC_ERR_TIMEOUT and carries on, so the launch
// always ends.
//
// Residual of the result (with_resid): P0 more units follow the K sweeps in
// the queue, one per diagonal-only level l.  The last sweep solved
// M z_K = N z_{K-1}, so Q^T z_K = N (z_{K-1} - z_K): zero on the coupled rows
// and T_lo d_{l-1} + T_up d_{l+1} (d = z_K - z_{K-1}) on the diagonal-only
// rows.  A residual unit waits until both neighbours hold z_K, reads z_K from
// Z and z_{K-1} from W (x_in when K = 1) and stores its level's L1 norm; this
// streams the off-diagonal blocks of half the levels once, a third of one
// sweep's bytes in inverse mode, instead of all three blocks of every level.
//
// Values and level sums do not depend on which team handles which unit, and
// the sums are reduced per level in a fixed order: results are bitwise
// reproducible for any grid.
#include <math.h>

#include "mc_internal.cuh"
#include "sweep_dev.cuh"
#include "team_dev.cuh"
#include "wave_dev.cuh"

namespace mc {

namespace {

using namespace dev;

// MC: the block size if it equals 32 RW TW, else 0.  BANDED: block-banded
// chains (Algorithm 2 with off-staircase terms, inverse mode): every row also
// adds sum_d T_{l,l+d} x_{l+d} over the far diagonals |d| >= 2 from the sweep's
// input, at levels of both parities, so the sweeps cannot update in place.
// Y_0 = x_in; sweep k reads Y_k and writes Y_{k+1} into W (k even) or Z (k
// odd), over Y_{k-1}.  A unit of sweep k at level l waits until every level
// within the band l - bw .. l + bw has finished sweep k - 1 (its inputs are
// ready and every reader of the Y_{k-1} it overwrites is done); a coupled-row
// unit also waits for half-sweep 1 of sweep k at l - 1 and l + 1.
//
// A level's completion counter grows by TW per write (each warp of the team
// releases its own rows).
template <int TW, int RW, int MC, bool COUPLED, bool PAIRED, bool BANDED>
__global__ void __launch_bounds__(TeamBlock<TW>::T, TeamBlock<TW>::B) k_sweeps(FusedArgs a) {
  extern __shared__ __align__(16) unsigned char team_smem[];
  using Sh = TeamShared<TW, RW>;
  static_assert(sizeof(Sh) % 16 == 0 && sizeof(TeamSlot<32 * RW * TW>) % 16 == 0, "pair loads");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int team = warp / TW, w = warp % TW, tt = threadIdx.x - team * TW * 32;
  Sh& sh = reinterpret_cast<Sh*>(team_smem)[team];
  const int bar = 1 + team;
  const int m = MC ? MC : a.m;
  const int row0 = 32 * RW * w;
  const unsigned long long sweeps = (unsigned long long)a.K * (unsigned long long)a.L;
  const unsigned long long total = sweeps + (a.with_resid ? (unsigned long long)a.P0 : 0ull);
  // paired chains: T_lo is zero in rows m/2.. of columns ..m/2, T_up in rows
  // ..m/2 of columns m/2.. (RW = 1: a warp's rows lie on one side)
  const int lo0 = PAIRED && 2 * row0 >= m ? m / 2 : 0;
  const int up1 = PAIRED && 2 * row0 < m ? m / 2 : m;
  int s = 0;   // ring position
  // one warp claims for the team; with one warp a unit ahead of use, with more
  // two ahead (the unit travels through shared memory with a barrier)
  unsigned long long q0 = w == 0 ? claim_unit(a.claim, lane) : 0ull, q;
  if constexpr (TW == 1) {
    q = __shfl_sync(kFull, q0, 0);
  } else {
    if (w == 0 && lane == 0) sh.next[1] = q0;
    if (w == 0) q0 = claim_unit(a.claim, lane);
    team_sync<TW>(bar);
    q = sh.next[1];
  }
  int turn = 0;
  while (q < total) {
    unsigned long long qn = 0ull;
    if constexpr (TW == 1) {
      q0 = claim_unit(a.claim, lane);   // its index is needed only after this unit
    } else if (w == 0 && lane == 0) {
      sh.next[turn] = q0;
    }
    const bool resid = !BANDED && q >= sweeps;
    const int64_t k = resid ? a.K : (int64_t)(q / (unsigned long long)a.L);
    const int64_t r = (int64_t)q - k * a.L;
    const bool h2 = !resid && r >= a.P0;
    const int64_t l = h2 ? 2 * (r - a.P0) + (1 - a.par0) : 2 * r + a.par0;
    const bool has_lo = l > 0, has_up = l < a.L - 1;
    const bool last = k == a.K - 1;
    double* dst = BANDED ? ((k & 1) ? a.Z : a.W) : (last ? a.Z : a.W);
    // half-sweep 1 reads z_k (x_in for k = 0); half-sweep 2 reads z_{k+1}; a
    // residual unit z_K and z_{K-1}
    const double* y = k == 0 ? a.x_in : (BANDED && !(k & 1)) ? a.Z : a.W;
    const double* src = resid ? a.Z : h2 ? dst : y;
    const int need = (int)(h2 ? k + 1 : k);
    // the blocks' exponents: loaded while this team waits
    const int2 none = make_int2(0, 0);
    const int2 ea = resid ? none : a.eA[l], eb = resid ? none : a.eB[l];
    const int2 ec = COUPLED || resid ? none : a.eC[l];
    if constexpr (BANDED) {
      if (need > 0)
        wait_band(a.ver, l, a.L, a.bw, (int)k * TW, need * TW, &a.hdr->status, lane, a.wait_ns);
    } else {
      if (need > 0) wait_neighbours(a.ver, l, a.L, need * TW, &a.hdr->status, lane, a.wait_ns);
    }
    // stage both neighbours: thread tt of the team loads rows tt, tt + 32 TW
    {
      double x0[RW], x1[RW];
#pragma unroll
      for (int i = 0; i < RW; ++i) {
        const int row = tt + 32 * TW * i;
        x0[i] = has_lo && row < m ? __ldcg(src + (l - 1) * m + row) : 0.0;
        x1[i] = has_up && row < m ? __ldcg(src + (l + 1) * m + row) : 0.0;
      }
      if (resid) {
#pragma unroll
        for (int i = 0; i < RW; ++i) {
          const int row = tt + 32 * TW * i;
          if (has_lo && row < m) x0[i] -= __ldcg(a.prev + (l - 1) * m + row);
          if (has_up && row < m) x1[i] -= __ldcg(a.prev + (l + 1) * m + row);
        }
      }
      stage_rows<RW>(sh.slot[s].v[0], sh.slot[s].x[0], sh.exps[s][0], x0, m, tt, 32 * TW, w, lane);
      stage_rows<RW>(sh.slot[s].v[1], sh.slot[s].x[1], sh.exps[s][1], x1, m, tt, 32 * TW, w, lane);
    }
    team_sync<TW>(bar);
    if constexpr (TW > 1) {
      qn = sh.next[turn];
      turn ^= 1;
      if (w == 0) q0 = claim_unit(a.claim, lane);
    }
    double acc[RW];
#pragma unroll
    for (int i = 0; i < RW; ++i) acc[i] = 0.0;
    if (resid) {
      // ||T_lo d_{l-1} + T_up d_{l+1}||_1, d = z_K - z_{K-1} (signed: FP64 pipe)
      if (has_lo)
        rows_f64<RW, MC>(acc, a.RA + (size_t)l * a.ms, sh.slot[s].v[0], lo0, m, m, row0, lane);
      if (has_up)
        rows_f64<RW, MC>(acc, a.RB + (size_t)l * a.ms, sh.slot[s].v[1], 0, up1, m, row0, lane);
      double t = 0.0;
#pragma unroll
      for (int i = 0; i < RW; ++i) t += fabs(acc[i]);
      t = team_total<TW>(warp_sum(t), sh.part, w, lane, bar);
      if (w == 0 && lane == 0) a.rsum[r] = t;
      s ^= 1;
      q = TW == 1 ? __shfl_sync(kFull, q0, 0) : qn;
      continue;
    }
    if (has_lo)
      rows_product<RW, MC>(acc, a.A + (size_t)l * a.ms, sh.slot[s].v[0], sh.slot[s].x[0], ea,
                           team_exp<TW>(sh.exps[s][0]), lo0, m, m, row0, lane);
    if (has_up)
      rows_product<RW, MC>(acc, a.B + (size_t)l * a.ms, sh.slot[s].v[1], sh.slot[s].x[1], eb,
                           team_exp<TW>(sh.exps[s][1]), 0, up1, m, row0, lane);
    if constexpr (BANDED) {
      const int n = a.far->n;
      for (int j = 0; j < n; ++j) {
        const int64_t kk = l + a.far->off[j];
        if (kk < 0 || kk >= a.L) continue;
        s ^= 1;
        const int2 ef = a.far->bexp[j][l];
        double x0[RW];
#pragma unroll
        for (int i = 0; i < RW; ++i) {
          const int row = tt + 32 * TW * i;
          x0[i] = row < m ? __ldcg(y + kk * m + row) : 0.0;
        }
        stage_rows<RW>(sh.slot[s].v[0], sh.slot[s].x[0], sh.exps[s][0], x0, m, tt, 32 * TW, w,
                       lane);
        team_sync<TW>(bar);
        rows_product<RW, MC>(acc, a.far->plane[j] + (size_t)l * a.ms, sh.slot[s].v[0],
                             sh.slot[s].x[0], ef, team_exp<TW>(sh.exps[s][0]), 0,
                             m, m, row0, lane);
      }
    }
    if constexpr (!COUPLED) {
      s ^= 1;
      stage_rows<RW>(sh.slot[s].v[0], sh.slot[s].x[0], sh.exps[s][0], acc, m, row0 + lane, 32, w,
                     lane);
      team_sync<TW>(bar);
#pragma unroll
      for (int i = 0; i < RW; ++i) acc[i] = 0.0;
      rows_product<RW, MC>(acc, a.C + (size_t)l * a.ms, sh.slot[s].v[0], sh.slot[s].x[0], ec,
                           team_exp<TW>(sh.exps[s][0]), 0, m, m, row0, lane);
    }
    double t = 0.0;
#pragma unroll
    for (int i = 0; i < RW; ++i) {
      const int row = row0 + lane + 32 * i;
      if (row < m) {
        dst[l * m + row] = acc[i];
        t += acc[i];
      }
    }
    __threadfence();
    __syncwarp();
    if (lane == 0) {
      if constexpr (TW == 1)
        st_release(a.ver + l, (int)(k + 1));
      else
        red_release(a.ver + l, 1);
    }
    // e^T z is needed of the last two sweeps only (FP64 adds cost issue slots)
    if (k >= a.K - 2) {
      t = team_total<TW>(warp_sum(t), sh.part, w, lane, bar);
      if (w == 0 && lane == 0) a.lsum[(k & 1) * a.L + l] = t;
    }
    s ^= 1;
    q = TW == 1 ? __shfl_sync(kFull, q0, 0) : qn;
  }
}

// Block Gauss-Seidel sweeps (Sect. 2 comparison splitting, M = block lower
// triangle of Q^T), all K sweeps of a call in one persistent launch:
// z^{k+1}_l = (-T_dd)^{-1} (T_lo z^{k+1}_{l-1} + T_up z^k_{l+1}) (inverse mode;
// W_lo, W_up when coupled).  Unit (k, l) needs (k, l-1) and (k-1, l+1), so the
// units are claimed in wavefront order (wave_unit): a sweep traverses the
// levels one after the other, each sweep trailing the previous one by two
// levels, and up to min(K, L / 2) units run at once.  In place in W (the
// last sweep writes Z): a unit overwrites z^k_l only after its two readers,
// (k, l-1) and (k-1, l+1), have completed, which is what it waits for.
//
// One block of kBgsWarps warps per unit: the warps split the columns of every
// block product (warp w takes a fixed even-aligned column range and keeps
// partial sums of all rows), and the partials are added in warp order.  A
// unit sits on the wavefront's critical path, so streaming its blocks with
// several warps' loads in flight instead of one shortens that path; the
// launch runs one block per unit in flight.  Four warps measured best (2, 4
// and 8 tried: fewer warps per unit leave more units resident at once).  Warp 0 waits for the two neighbours, the block barrier
// hands the wait on (every warp also acquires both counters), and after its
// stores every thread fences before thread 0 releases the level.  The
// vectors sit in block shared memory with 16 zero doubles of padding, so a
// warp's last column batch may read past its range (those products are with
// zero block entries).
constexpr int kBgsWarps = 4;

__device__ __forceinline__ double bgs_parts(const double* part, int W, int i) {
  static_assert(kBgsWarps == 4, "");
  return (part[i] + part[W + i]) + (part[2 * W + i] + part[3 * W + i]);
}

template <int R, bool COUPLED>
__global__ void __launch_bounds__(32 * kBgsWarps, 16 / kBgsWarps) k_bgs_cta(FusedArgs a) {
  constexpr int W = 32 * R, VS = W + 16;
  extern __shared__ double sh[];
  double* v_lo = sh;
  double* v_up = sh + VS;
  double* v_g = sh + 2 * VS;
  double* part = sh + 3 * VS;   // kBgsWarps x W partial sums
  __shared__ double red[kBgsWarps];
  __shared__ unsigned long long s_q;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nt = blockDim.x;
  const int m = a.m;
  const int cw = (((m + kBgsWarps - 1) / kBgsWarps) + 1) & ~1;
  const int j0 = w * cw, j1 = j0 + cw < m ? j0 + cw : m;
  for (int i = threadIdx.x; i < 3 * VS; i += nt) sh[i] = 0.0;   // pads stay zero
  const unsigned long long total = (unsigned long long)a.K * (unsigned long long)a.L;
  while (true) {
    if (threadIdx.x == 0) s_q = atomicAdd(a.claim, 1ull);
    __syncthreads();
    const unsigned long long q = s_q;
    if (q >= total) break;
    int64_t k, l;
    wave_unit(q, a.L, a.K, &k, &l);
    double* dst = k == a.K - 1 ? a.Z : a.W;
    const double* up = k == 0 ? a.x_in : a.W;    // z^k at l + 1
    const bool has_lo = l > 0, has_up = l < a.L - 1;
    if (w == 0)
      wait_neighbours2(a.ver, l, a.L, (int)(k + 1), (int)k, &a.hdr->status, lane, a.wait_ns);
    __syncthreads();
    if (w != 0) {
      if (has_lo) (void)ld_acquire(a.ver + l - 1);
      if (has_up && k > 0) (void)ld_acquire(a.ver + l + 1);
    }
    for (int i = threadIdx.x; i < m; i += nt) {
      v_lo[i] = has_lo ? __ldcg(dst + (l - 1) * m + i) : 0.0;
      v_up[i] = has_up ? __ldcg(up + (l + 1) * m + i) : 0.0;
    }
    __syncthreads();
    double acc[R];
    zero_acc<R>(acc);
    if (j0 < j1) {
      if (has_lo) gemv_acc<R>(acc, a.A + (size_t)l * a.ms, v_lo, j0, j1, m, lane);
      if (has_up) gemv_acc<R>(acc, a.B + (size_t)l * a.ms, v_up, j0, j1, m, lane);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) part[w * W + lane + 32 * r] = acc[r];
    __syncthreads();
    if (!COUPLED) {
      for (int i = threadIdx.x; i < m; i += nt) v_g[i] = bgs_parts(part, W, i);
      __syncthreads();
      zero_acc<R>(acc);
      if (j0 < j1) gemv_acc<R>(acc, a.C + (size_t)l * a.ms, v_g, j0, j1, m, lane);
#pragma unroll
      for (int r = 0; r < R; ++r) part[w * W + lane + 32 * r] = acc[r];
      __syncthreads();
    }
    double ls = 0.0;
    for (int i = threadIdx.x; i < m; i += nt) {
      const double z = bgs_parts(part, W, i);
      dst[l * m + i] = z;
      ls += z;
    }
    if (k >= a.K - 2) {   // e^T z of the last two sweeps only (uniform over the block)
      ls = block_sum(ls, red);
      if (threadIdx.x == 0) a.lsum[(k & 1) * a.L + l] = ls;
    }
    __threadfence();
    __syncthreads();   // every store of z_l, and every read of part, before the release
    if (threadIdx.x == 0) st_release(a.ver + l, (int)(k + 1));
  }
}

// Self-test of the bounded wait: one warp waits for level 1 of a 3-level
// counter array; the counters hold `preset`, the wait needs 1.
__global__ void k_wait_selftest(int preset, unsigned long long wait_ns, Header* hdr, int* ver) {
  const int lane = threadIdx.x & 31;
  if (lane < 3) ver[lane] = preset;
  __syncwarp();
  wait_neighbours(ver, 1, 3, 1, &hdr->status, lane, wait_ns);
}

// e^T z_K and e^T z_{K-1} from the per-level sums, and the residual from the
// per-level residual norms.  FP64 adds run at two lanes per clock per SM
// here, so the sums are spread over kScaleBlocks blocks, each over a fixed
// contiguous range of levels; the last block to finish adds the block
// partials (fixed summation order).
// part: 3 kScaleBlocks doubles of scratch; ticket: zero between launches.
__global__ void __launch_bounds__(256) k_fused_scale(const double* lsum, int64_t L, int64_t K,
                                                     const double* rsum, int64_t P,
                                                     double* part, unsigned* ticket,
                                                     double* out) {
  __shared__ double sh[32];
  __shared__ bool last;
  const double* a = lsum + ((K - 1) & 1) * L;
  const double* b = lsum + ((K - 2) & 1) * L;
  const int64_t chunk = (L + gridDim.x - 1) / gridDim.x;
  const int64_t l0 = blockIdx.x * chunk;
  const int64_t l1 = l0 + chunk < L ? l0 + chunk : L;
  double ta = 0.0, tb = 0.0, tr = 0.0;
  for (int64_t l = l0 + threadIdx.x; l < l1; l += blockDim.x) {
    ta += a[l];
    if (K >= 2) tb += b[l];
  }
  if (rsum) {
    const int64_t pc = (P + gridDim.x - 1) / gridDim.x;
    const int64_t p0 = blockIdx.x * pc;
    const int64_t p1 = p0 + pc < P ? p0 + pc : P;
    for (int64_t u = p0 + threadIdx.x; u < p1; u += blockDim.x) tr += rsum[u];
  }
  ta = block_sum0(ta, sh);
  if (K >= 2) tb = block_sum0(tb, sh);
  if (rsum) tr = block_sum0(tr, sh);
  if (threadIdx.x == 0) {
    part[3 * blockIdx.x] = ta;
    part[3 * blockIdx.x + 1] = tb;
    part[3 * blockIdx.x + 2] = tr;
    __threadfence();
    last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last || threadIdx.x >= 32) return;
  __threadfence();
  // the first warp loads the partials in parallel (lane i: blocks i, i + 32)
  // and adds them with a fixed shuffle tree
  double sa = 0.0, sb = 0.0, sr = 0.0;
  for (int i = threadIdx.x; i < (int)gridDim.x; i += 32) {
    sa += __ldcg(part + 3 * i);
    sb += __ldcg(part + 3 * i + 1);
    sr += __ldcg(part + 3 * i + 2);
  }
  sa = warp_sum(sa);
  sb = warp_sum(sb);
  sr = warp_sum(sr);
  if (threadIdx.x == 0) {
    out[0] = sa;
    out[1] = K >= 2 ? sb : 1.0;
    out[2] = rsum ? sr : nan("");
    *ticket = 0u;
  }
}

// bps: resident blocks per SM (0: all the kernel's occupancy allows); no more
// teams than levels.
template <int TW, int RW, int MC, bool C, bool P, bool BANDED>
cudaError_t sweeps_k(const FusedArgs& a, int bps, int sms, cudaStream_t s) {
  constexpr int T = TeamBlock<TW>::T, teams = T / 32 / TW;
  static int occ = 0;
  const size_t smem = teams * sizeof(TeamShared<TW, RW>);
  if (occ == 0) {
    cudaError_t e = cudaFuncSetAttribute(k_sweeps<TW, RW, MC, C, P, BANDED>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int o = 0;
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_sweeps<TW, RW, MC, C, P, BANDED>, T,
                                                        smem);
    if (e != cudaSuccess) return e;
    occ = o < 1 ? 1 : o;
  }
  int64_t nb = (int64_t)(bps > 0 && bps < occ ? bps : occ) * sms;
  const int64_t need = (a.L + teams - 1) / teams;
  if (nb > need) nb = need;
  k_sweeps<TW, RW, MC, C, P, BANDED><<<(int)nb, T, smem, s>>>(a);
  return cudaGetLastError();
}

template <int TW, int RW, bool C, bool P, bool BANDED>
cudaError_t sweeps_m(const FusedArgs& a, int bps, int sms, cudaStream_t s) {
  if constexpr (P)
    return sweeps_k<TW, RW, 32 * RW * TW, C, P, BANDED>(a, bps, sms, s);
  else
    return a.m == 32 * RW * TW ? sweeps_k<TW, RW, 32 * RW * TW, C, P, BANDED>(a, bps, sms, s)
                               : sweeps_k<TW, RW, 0, C, P, BANDED>(a, bps, sms, s);
}

// Team of a block size: two rows per lane (half the warps per level, so half
// the staging and waiting per streamed byte) while a half-sweep has more units
// than teams in flight; one row per lane (twice the warps per level) when it
// has fewer, so that units neither wait for their neighbours' previous sweep
// nor leave warps without work.
template <bool C, bool BANDED>
cudaError_t sweeps_team(const FusedArgs& a, int bps, int sms, cudaStream_t s) {
  const int r = (a.m + 31) / 32;
  const int64_t teams2 = 24ll * sms / ((r + 1) / 2);
  const bool narrow = r == 1 || a.L / 2 < teams2 + teams2 / 2;
  if (narrow) {
    switch (r) {
      case 1: return sweeps_m<1, 1, C, false, BANDED>(a, bps, sms, s);
      case 2: return sweeps_m<2, 1, C, false, BANDED>(a, bps, sms, s);
      case 3:
      case 4: return sweeps_m<4, 1, C, false, BANDED>(a, bps, sms, s);
      case 5:
      case 6: return sweeps_m<6, 1, C, false, BANDED>(a, bps, sms, s);
      default: return sweeps_m<8, 1, C, false, BANDED>(a, bps, sms, s);
    }
  }
  switch ((r + 1) / 2) {
    case 1: return sweeps_m<1, 2, C, false, BANDED>(a, bps, sms, s);
    case 2: return sweeps_m<2, 2, C, false, BANDED>(a, bps, sms, s);
    case 3: return sweeps_m<3, 2, C, false, BANDED>(a, bps, sms, s);
    default: return sweeps_m<4, 2, C, false, BANDED>(a, bps, sms, s);
  }
}

// nb: units that can run at once (capped here at the blocks resident at once,
// so every claimed unit belongs to a running block).
template <int R, bool C>
cudaError_t bgs_fused_r(const FusedArgs& a, int nb, cudaStream_t s) {
  static int cap = 0;
  const size_t smem = (size_t)(3 * (32 * R + 16) + kBgsWarps * 32 * R) * sizeof(double);
  if (cap == 0) {
    int dev = 0, sms = 0, occ = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_bgs_cta<R, C>, 32 * kBgsWarps,
                                                        smem);
    if (e != cudaSuccess) return e;
    cap = (occ < 1 ? 1 : occ) * sms;
  }
  if (nb > cap) nb = cap;
  if (nb < 1) nb = 1;
  k_bgs_cta<R, C><<<nb, 32 * kBgsWarps, smem, s>>>(a);
  return cudaGetLastError();
}

template <bool C>
cudaError_t sweeps_dispatch(const FusedArgs& a, int bps, int sms, cudaStream_t s) {
  if (a.m < 1 || a.m > kMaxM) return cudaErrorInvalidValue;
  if (a.bgs) {
    if (a.far || a.paired) return cudaErrorInvalidValue;
    // at most min(K, L/2) units run at once (one per sweep in flight), one
    // block per unit; the launcher caps the grid at the blocks resident at once
    const int64_t par = a.K < (a.L + 1) / 2 ? a.K : (a.L + 1) / 2;
    int nb = par < (1 << 30) ? (int)par : (1 << 30);
    if (bps > 0 && bps * sms < nb) nb = bps * sms;
    switch ((a.m + 31) / 32) {
      case 1: return bgs_fused_r<1, C>(a, nb, s);
      case 2: return bgs_fused_r<2, C>(a, nb, s);
      case 3: return bgs_fused_r<3, C>(a, nb, s);
      case 4: return bgs_fused_r<4, C>(a, nb, s);
      case 5: return bgs_fused_r<5, C>(a, nb, s);
      case 6: return bgs_fused_r<6, C>(a, nb, s);
      case 7: return bgs_fused_r<7, C>(a, nb, s);
      default: return bgs_fused_r<8, C>(a, nb, s);
    }
  }
  if (a.far) {
    if constexpr (C)
      return cudaErrorInvalidValue;   // block-banded chains: inverse mode only
    else
      return sweeps_team<false, true>(a, bps, sms, s);
  }
  if (a.paired && !C) {
    switch (a.m / 32) {
      case 2: return sweeps_m<2, 1, false, true, false>(a, bps, sms, s);
      case 4: return sweeps_m<4, 1, false, true, false>(a, bps, sms, s);
      case 6: return sweeps_m<6, 1, false, true, false>(a, bps, sms, s);
      case 8: return sweeps_m<8, 1, false, true, false>(a, bps, sms, s);
      default: return cudaErrorInvalidValue;
    }
  }
  return sweeps_team<C, false>(a, bps, sms, s);
}

}  // namespace

cudaError_t launch_sweeps_fused(const FusedArgs& a, int coupled, int bps, int sms,
                                cudaStream_t s) {
  return coupled ? sweeps_dispatch<true>(a, bps, sms, s) : sweeps_dispatch<false>(a, bps, sms, s);
}

cudaError_t launch_wait_selftest(int preset, unsigned long long wait_ns, Header* hdr, int* ver,
                                 cudaStream_t s) {
  k_wait_selftest<<<1, 32, 0, s>>>(preset, wait_ns, hdr, ver);
  return cudaGetLastError();
}

cudaError_t launch_fused_scale(const double* lsum, int64_t L, int64_t K, const double* rsum,
                               int64_t P, double* out, double* part, unsigned* ticket,
                               cudaStream_t s) {
  k_fused_scale<<<kScaleBlocks, 256, 0, s>>>(lsum, L, K, rsum, P, part, ticket, out);
  return cudaGetLastError();
}

}  // namespace mc

namespace {
struct WaitSelftestScratch {
  mc::Header hdr;
  int ver[4];
};
__device__ __align__(256) WaitSelftestScratch g_wait_selftest;
}  // namespace

extern "C" int mc_wait_selftest(void* cuda_stream, int reachable, int64_t wait_ns) {
  if (wait_ns < 0 || wait_ns > 10000000000ll) return MC_ERR_ARG;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  void* p = nullptr;
  if (cudaGetSymbolAddress(&p, g_wait_selftest) != cudaSuccess || !p) return MC_ERR_CUDA;
  WaitSelftestScratch* w = (WaitSelftestScratch*)p;
  if (cudaMemsetAsync(w, 0, sizeof(WaitSelftestScratch), s) != cudaSuccess) return MC_ERR_CUDA;
  if (mc::launch_wait_selftest(reachable ? 1 : 0, (unsigned long long)wait_ns, &w->hdr, w->ver,
                               s) != cudaSuccess)
    return MC_ERR_CUDA;
  int status = 0;
  if (cudaMemcpyAsync(&status, &w->hdr.status, sizeof(int), cudaMemcpyDeviceToHost, s) !=
          cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return MC_ERR_CUDA;
  return status;
}
