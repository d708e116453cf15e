// Batched (multi-request) sweep: descriptors shared by batch.cu and server.cu.
//
// All active requests of the solve server advance together: fused persistent
// launches side by side cover every level of every request for all sweeps of
// a chunk, by path (below).  The request table lives in device memory and is
// rewritten by the host between chunks, so one captured CUDA graph serves any
// active set that uses the same launches.  Requests are ordered by size class
// (m <= 32, m <= 64, m <= 128, m <= 256).  On the low-precision queue a bucket
// is a run of classes launched as one kernel sized for its largest block, so
// that register use follows the bucket; where the bucket edges lie is a tuning
// choice (BTune::split64).
//
// Every reduction is per level first (one partial per level), then per
// request in level order: a request's iterates do not depend on which other
// requests share the launch, nor on any choice of the autotuner (grid,
// levels per unit, bucket edges, load depth).
//
// The sweeps of a chunk run fused (as the single-chain fused sweeps): all of
// them in one persistent launch, units claimed in order, each waiting for its
// neighbour levels through the request's completion counters.  On the queue a
// unit covers G adjacent levels of one half-sweep of
// one request (levels l0, l0 + 2, ..., l0 + 2 (G - 1); G per request, from
// the table's G and the request's size class): one claim, one wait for the
// G + 1 neighbour levels, one completion fence.  Counters grow across
// chunks: a chunk with epoch E writes E + k + 1 after its sweep k, so counters
// never need resetting (new requests start at zero <= E); the claim counters
// live in the table and are reset by the table copy that starts every chunk.
#pragma once
#include "mc_internal.cuh"

namespace mc {

constexpr int kMaxReq = 1024;

struct BReq {
  const double* A;      // FP64 sweep operators: T_lo / W_lo
  const double* B;      // T_up / W_up
  const double* C;      // (-T_dd)^{-1} (inverse mode)
  const double* TLO;    // residual blocks
  const double* TDD;
  const double* TUP;
  const double* NINV;
  const void* lA;       // low-precision operators (dtype MC_F32 / MC_BF16)
  const void* lB;
  const float* lC;
  const float* sc;
  float* d;             // correction (low precision)
  float* q;             // (-T_dd)^{-1} r
  double* x;            // iterate pi
  double* z;            // unnormalised sweep output
  double* xb;           // pi + d before renormalisation
  double* lsum;         // one partial per level
  double* lsum2;        // fused sweeps: [2][L] level sums of the last two sweeps
  int* ver;             // fused sweeps: per-level completion counters
  int64_t L;
  unsigned long long* dv;   // low precision: versioned words of the correction (team path)
  const int2* eA;       // FP64: block_exp of A, B, C (team path)
  const int2* eB;
  const int2* eC;
  int32_t m, ms, smem, p1;  // smem: shared memory of a CTA of the resident path; p1: 0-based
                            // parity of the diagonal-only rows
  int32_t G, path;       // levels per unit of this request (the table's G scaled by size
                         // class); kPathQueue, ...
  int32_t vbase;         // FP64 team path: sweeps that the counters have seen
  int16_t res_c, res_s;  // FP64 queue: CTAs of the cluster whose order of sums applies (0:
                         // columns in order) and its column groups (0: by the level)
  int64_t lp_bs, lp_cbs;
};

// Size classes of the request table: m <= 32, 64, 128, 256.
constexpr int kClasses = 4;
__host__ __device__ inline int size_class(int m) { return m <= 32 ? 0 : m <= 64 ? 1 : m <= 128 ? 2 : 3; }
// Levels per unit of a request: the table's G times 4, 2, 1, 1 by size class
// (at most 16), so that a unit of small blocks carries about as many bytes as
// one of m <= 128 and the claim, the wait and the fence are paid less often.
__host__ __device__ inline int class_group(int G, int m) {
  const int c = size_class(m);
  const int g = G * (c == 0 ? 4 : c == 1 ? 2 : 1);
  return g > 16 ? 16 : g;
}

// How a request's sweeps run.  Its arithmetic follows from its own size alone (so that
// its iterates do not depend on the batch):
//   kPathQueue: one warp per unit of G levels, all such requests in shared launches
//     by size class (k_b_sweeps, k_b_sweeps_lp);
//   kPathTeam: a team of warps per level, all such requests of a size class in one
//     launch: FP64 requests (team_dev.cuh), low-precision short chains of blocks of
//     more than 32 rows (lpteam_dev.cuh);
//   kPathResident: blocks of up to 32 rows that fit one cluster's shared memory, one
//     cluster per request (resident_dev.cuh).
// FP64 requests of the resident path run on the queue, with the sums in the resident
// order (res_c), while so many are active that the clusters would take longer, and
// FP64 blocks of up to 16 rows of the team path, which adds as the queue does, while
// their levels fill the GPU several times over (build_table).
// The launches of the three paths run side by side; the host deals out CTAs to
// them with the table.  Eight requests of 131 KB to 17 MB
// (BF16 coupled, m = 16 to 128): a chunk of 64 sweeps 2.70 -> 0.99 ms with all of them
// running, 1.32 -> 0.24 ms with the last two small ones.
enum { kPathQueue = 0, kPathTeam = 1, kPathResident = 2 };
// One bit per path and size class (queue: 0) or resident group.
inline int path_bit(int path, int cls) { return 1 << (5 * path + cls); }

// Resident requests by group, a launch each.  A cluster alone leaves most of its SMs'
// time to latency, so a batch of many small low-precision requests needs several
// clusters on the same SMs: a group is a number of CTAs that share an SM, given by
// their shared memory and by the registers of the kernel (blocks of up to 16 rows hold
// their operators in registers, wider ones, `wide`, do not).  A chunk of 64 sweeps,
// one CTA an SM -> shared (the queue): 250 of 128 x 16, BF16 coupled, 2.97 -> 1.61 ms
// (2.15); 200 of 90 x 24, FP32 inverse, 7.3 -> 1.76 (2.81); 100 of 400 x 20, BF16
// coupled, 3.18 -> 1.12 (3.97).  What fits an SM only once is as before: below the
// queue's rate where 60 or more of FP32 or inverse mode with m > 16 run at once (100
// of 200 x 28, FP32 inverse: 4.1, queue 2.7), far above it where few do (one of
// 300 x 32: 0.20, queue 1.27).
constexpr int kResGroups = 5;
constexpr int kResidentSlots = 8;      // sets of 16 SMs given to clusters
__host__ __device__ constexpr int group_share(int group) {
  return group == 0 ? 2 : group == 2 ? 4 : group == 3 ? 2 : 1;
}
__host__ __device__ constexpr bool group_wide(int group) { return group == 2 || group == 3; }

struct BTable {
  int32_t n;            // active requests, ordered by size class
  int32_t cls_end[kClasses];     // requests [0, cls_end[c]) have size class <= c
  int32_t epoch;        // completion-counter base of this chunk
  int32_t G;            // levels per unit of the fused sweep launches (1, 2 or 4), scaled
                        // per request by class_group
  int32_t res_end[kResGroups];        // resident requests of the groups up to this one
  int32_t res_clusters[kResGroups];   // and the clusters that take a group's
  int32_t team_ctas[kClasses];   // CTAs of the team launch of a size class
  // (the counters on lines of their own: next to the offsets that every unit reads a
  // chunk of three chains of 6000 levels took 1.48 ms instead of 1.42)
  alignas(128) unsigned long long claim[kClasses];   // queue counters of one chunk's buckets (0 in t_host)
  alignas(128) int64_t off_h1[kMaxReq + 1];   // prefix counts of half-sweep-1 units (groups of G levels)
  int64_t off_h2[kMaxReq + 1];   // prefix counts of half-sweep-2 units
  int64_t off_lv[kMaxReq + 1];   // prefix counts of all levels
  alignas(128) unsigned long long team_claim[kClasses];   // queue counters of the team launches
  alignas(128) int64_t off_t1[kMaxReq + 1];   // prefix counts of the team path's levels by half-sweep
  int64_t off_t2[kMaxReq + 1];
  int32_t res[kMaxReq];          // table positions of the resident requests, by group
  BReq r[kMaxReq];
};

struct BOut {
  double s, step, resid;
  double s_last, s_prev;   // fused FP64 chunk: e^T z of its last two sweeps (s_prev = 1 for one)
  int32_t status;
  int32_t pad;
};

// Launch configuration of a chunk, chosen per batch signature by the server's
// autotuner from live chunk timings.  The levels per unit G travel in the
// request table (its unit prefix counts depend on G).
struct BTune {
  int blocks, threads;  // persistent grid of the fused launches
  int split64;          // low precision: 1: m <= 64 in a launch of its own,
                        // 0: m <= 128 in one launch
  int deep;             // low-precision blocks of m <= 64: 16 (1) or 8 (0) loads in flight
};

// The buckets (runs of size classes launched as one kernel) of a tuning of the
// low-precision queue, [c0[i], c1[i]) for i < n.
struct BBuckets {
  int n;
  int c0[kClasses], c1[kClasses];
};
inline BBuckets buckets_of(int split64) {
  BBuckets b{};
  if (split64) {
    b.n = 3;
    b.c0[0] = 0, b.c1[0] = 2;
    b.c0[1] = 2, b.c1[1] = 3;
    b.c0[2] = 3, b.c1[2] = 4;
  } else {
    b.n = 2;
    b.c0[0] = 0, b.c1[0] = 3;
    b.c0[1] = 3, b.c1[1] = 4;
  }
  return b;
}

// After K FP64 sweeps of every request: e^T z, normalisation and the step error
// of the last sweep.
cudaError_t b_sweeps_finish(const BTable* t, BOut* out, int K, BTune g, cudaStream_t s);
// Direct residual of every request's iterate (with_q: also q for refinement).
cudaError_t b_resid(const BTable* t, BOut* out, int with_q, BTune g, cudaStream_t s);
// Mixed precision: d = 0 (b_lp_zero; queue path only, the others write d once);
// `inner` fused correction sweeps (b_lp_sweeps; t_claim: the device table's claim counters; coupled: server-wide
// apply mode); pi <- (pi + d)/e^T(pi + d) with the step error (b_lp_finish).
cudaError_t b_lp_zero(const BTable* t, BTune g, cudaStream_t s);
cudaError_t b_lp_sweeps(const BTable* t, unsigned long long* t_claim, BOut* out, int bf16,
                        int coupled, int inner, BTune g, cudaStream_t s);
// The team requests' correction sweeps, a launch per size class on b0, b[0..2].
// paths: the path_bit of every path and size class of the table.
cudaError_t b_lp_team(const BTable* t, unsigned long long* team_claim, BOut* out, int paths,
                      int bf16, int coupled, int inner, int num_sms, const cudaStream_t* b);
// Path of a request of this layout.
int b_path(const Layout& lay, int coupled, int num_sms);
// The FP64 queue's sweeps.
cudaError_t b_sweeps(const BTable* t, unsigned long long* claim, BOut* out, int coupled, int K,
                     BTune g, cudaStream_t s);
// The FP64 team requests' sweeps, a launch per size class on b0, b[0..2].
cudaError_t b_team(const BTable* t, unsigned long long* team_claim, BOut* out, int paths,
                   int coupled, int K, int num_sms, cudaStream_t b0, const cudaStream_t* b);
// resident.cu: CTAs of a cluster (0: none can run); the group of a request that fits
// one cluster, else -1, and a CTA's shared memory; res_c and res_s of an FP64 request;
// the launch of a group's requests (lp: 0 FP64, 1 FP32, 2 BF16).
int resident_cluster();
int resident_batch_group(const Layout& lay, int coupled);
int resident_batch_smem(const Layout& lay, int coupled);
cudaError_t launch_resident_batch(const BTable* t, int lp, int coupled, int group, int K, BOut* out,
                                  cudaStream_t s);
void resident_order(const Layout& lay, int16_t* c, int16_t* s);
cudaError_t b_lp_finish(const BTable* t, BOut* out, BTune g, cudaStream_t s);

}  // namespace mc
