// Continuous-batching solve server (C ABI in include/mc.h, mc_server_*).
//
// Requests (independent chains of any L and m <= 256) are admitted into a
// caller-owned device arena as long as their workspace fits; each step runs
// one chunk of check_every sweeps for ALL active requests with the batched
// kernels of batch.cu and resident.cu (fused persistent launches side by side,
// by path: batch.cuh), then reads every request's residual and retires the converged
// ones.  New requests join at the next chunk, so their work overlaps with the
// requests already running.  A chunk is one CUDA graph, captured once per
// (grid, chunk length, launches in use) and replayed: the kernels read the request table from
// device memory, which the graph itself refreshes from pinned host memory.
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <deque>
#include <map>
#include <new>
#include <vector>

#include "batch.cuh"
#include "chain.cuh"
#include "deal.h"

using namespace mc;

namespace {

constexpr size_t kAlign = 256;

size_t align_up(size_t v) { return (v + kAlign - 1) / kAlign * kAlign; }

struct Req {
  int64_t tag;
  mc_chain* chain;
  size_t off, bytes;
  double* lsum;
  int64_t sweeps;
  double step_prev;
  int path;             // kPathQueue / kPathTeam / kPathResident
  int group;            // of the resident path
  int64_t vbase;        // value of the completion counters per warp of a level's team (FP64)
  bool fresh;           // factor status not yet checked
};

constexpr int kSides = kResGroups + kClasses - 1;

struct Done {
  int64_t tag;
  double* pi;           // host copy of the result (malloc), N doubles
  int64_t N;
  mc_result res;
  int status;
};

}  // namespace

struct mc_server {
  mc_server_desc d;
  char* arena;
  size_t arena_bytes;
  cudaStream_t user;
  int num_sms;
  std::map<size_t, size_t> free_;   // offset -> size, coalesced
  BTable* t_dev;
  BOut* out_dev;
  BTable* t_host;                   // pinned
  BOut* out_host;                   // pinned
  std::vector<Req*> active;
  std::deque<Done> done;
  cudaStream_t cap;
  cudaStream_t side[kSides];        // resident groups and team classes run beside the others
  cudaEvent_t fork[2], join[kSides];
  cudaGraphExec_t gexec;
  BTune g_tune;          // configuration of the captured graph
  int g_chunk;
  int g_paths;           // table_paths of the captured graph
  int G;                 // levels per unit of the table being built
  std::map<uint64_t, BTune> tuned;
  std::map<uint64_t, int> tuned_G;
  // autotuner results: (signature, candidate, ms per chunk) of every timed chunk
  std::vector<mc_server_tuning> trials;
  int64_t chunks;
  int32_t epoch_next;   // completion-counter base of the next chunk
};

namespace {

bool alloc(mc_server* s, size_t bytes, size_t* off) {
  for (auto it = s->free_.begin(); it != s->free_.end(); ++it) {
    if (it->second >= bytes) {
      *off = it->first;
      const size_t rest = it->second - bytes;
      const size_t start = it->first + bytes;
      s->free_.erase(it);
      if (rest) s->free_[start] = rest;
      return true;
    }
  }
  return false;
}

void release(mc_server* s, size_t off, size_t bytes) {
  auto it = s->free_.emplace(off, bytes).first;
  auto nx = std::next(it);
  if (nx != s->free_.end() && it->first + it->second == nx->first) {
    it->second += nx->second;
    s->free_.erase(nx);
  }
  if (it != s->free_.begin()) {
    auto pv = std::prev(it);
    if (pv->first + pv->second == it->first) {
      pv->second += it->second;
      s->free_.erase(it);
    }
  }
}

mc_desc request_desc(const mc_server* s, int64_t L, int32_t m) {
  mc_desc d{};
  d.L = L;
  d.m = m;
  d.stair = s->d.stair;
  d.apply = s->d.apply;
  d.dtype = s->d.dtype;
  return d;
}

size_t request_bytes(const mc_server* s, int64_t L, int32_t m) {
  const mc_desc d = request_desc(s, L, m);
  const size_t ws = mc_workspace_bytes(&d);
  if (!ws) return 0;
  return align_up(ws) + align_up((size_t)L * sizeof(double));
}

void fill_req(const mc_server* s, const Req* r, BReq* q) {
  mc_chain* c = r->chain;
  const size_t pe = c->lay.plane_bytes / sizeof(double);
  const bool coupled = s->d.apply == MC_APPLY_COUPLED;
  memset(q, 0, sizeof(*q));
  q->A = c->planes + (coupled ? kPlaneWLO : kPlaneTLO) * pe;
  q->B = c->planes + (coupled ? kPlaneWUP : kPlaneTUP) * pe;
  q->C = c->planes + kPlaneNINV * pe;
  q->TLO = c->planes + kPlaneTLO * pe;
  q->TDD = c->planes + kPlaneTDD * pe;
  q->TUP = c->planes + kPlaneTUP * pe;
  q->NINV = c->planes + kPlaneNINV * pe;
  q->eA = chain_bexp(c, coupled ? kPlaneWLO : kPlaneTLO);
  q->eB = chain_bexp(c, coupled ? kPlaneWUP : kPlaneTUP);
  q->eC = chain_bexp(c, kPlaneNINV);
  q->vbase = (int32_t)r->vbase;
  if (c->lay.lp) {
    q->lA = chain_lpA(c);
    q->lB = chain_lpB(c);
    q->lC = chain_lpC(c);
    q->sc = chain_lpSc(c);
    q->d = chain_lpD(c);
    q->dv = (unsigned long long*)c->z;   // FP64 sweeps only write z
    q->q = chain_lpQ(c);
    q->lp_bs = c->lay.lp_bs;
    q->lp_cbs = c->lay.lp_cbs;
  }
  q->x = c->xa;
  q->z = c->z;
  q->xb = c->xb;
  q->lsum = r->lsum;
  q->lsum2 = c->flsum;
  q->ver = c->fver;
  q->L = c->lay.L;
  q->m = c->lay.m;
  q->ms = c->lay.ms;
  if (r->path == kPathResident) q->smem = resident_batch_smem(c->lay, coupled);
  q->p1 = s->d.stair == 1 ? 0 : 1;
  q->path = r->path;
}

// Retire request i of the active list: copy pi to the host, free its memory.
int retire(mc_server* s, size_t i, int status, double resid, double step, double kappa,
           int converged) {
  Req* r = s->active[i];
  Done dn{};
  dn.tag = r->tag;
  dn.N = r->chain->lay.N;
  dn.status = status;
  dn.pi = (double*)malloc(sizeof(double) * (size_t)dn.N);
  int rc = MC_OK;
  if (!dn.pi) rc = MC_ERR_ARG;
  if (rc == MC_OK && cudaMemcpy(dn.pi, r->chain->xa, sizeof(double) * (size_t)dn.N,
                                cudaMemcpyDeviceToHost) != cudaSuccess)
    rc = MC_ERR_CUDA;
  dn.res.sweeps = r->sweeps;
  dn.res.residual_l1 = resid;
  dn.res.step_l1 = step;
  dn.res.contraction = kappa;
  dn.res.converged = converged;
  // a result that could not be copied out is reported as failed, without pi
  if (rc != MC_OK) {
    free(dn.pi);
    dn.pi = nullptr;
    if (dn.status == MC_OK) dn.status = rc;
    dn.res.converged = 0;
  }
  s->done.push_back(dn);
  mc_destroy(r->chain);
  release(s, r->off, r->bytes);
  delete r;
  s->active.erase(s->active.begin() + (long)i);
  return rc;
}

// The words of a team-path request to version 0.
cudaError_t reset_team_words(mc_server* s, const Req* r) {
  if (r->path != kPathTeam || !r->chain->lay.lp) return cudaSuccess;
  return cudaMemsetAsync(r->chain->z, 0, (size_t)r->chain->lay.N * sizeof(unsigned long long),
                         s->user);
}

// The next chunk (about to run) uses the current counter base; the one after
// it starts c higher.  Called before each execution of a chunk (a direct
// enqueue or a graph launch), while no chunk is in flight.  Before the 32-bit
// counters could wrap, every active request's counters are zeroed (stream
// ordered before the chunk) and the base restarts at 0.
int begin_chunk(mc_server* s, int c) {
  if (s->epoch_next > (1 << 27)) {   // the teams' counters advance by up to 8 a sweep
    for (size_t i = 0; i < s->active.size(); ++i) {
      Req* r = s->active[i];
      r->vbase = 0;
      s->t_host->r[i].vbase = 0;   // the table is in the order of the active list
      if (cudaMemsetAsync(r->chain->fver, 0, (size_t)r->chain->lay.L * sizeof(int), s->user) !=
              cudaSuccess ||
          reset_team_words(s, r) != cudaSuccess)
        return MC_ERR_CUDA;
    }
    s->epoch_next = 0;
  }
  s->t_host->epoch = s->epoch_next;
  s->epoch_next += c;
  return MC_OK;
}

// The paths, team size classes and resident groups that the table's requests use.
int table_paths(const BTable* t) {
  int p = 0;
  for (int i = 0; i < t->n; ++i)
    if (t->r[i].path != kPathResident)
      p |= path_bit(t->r[i].path, t->r[i].path == kPathTeam ? size_class(t->r[i].m) : 0);
  for (int g = 0; g < kResGroups; ++g)
    if (t->res_end[g] > (g ? t->res_end[g - 1] : 0)) p |= path_bit(kPathResident, g);
  return p;
}

// Chunk body on stream st: c fused sweeps (FP64) or one refinement step of c
// fused correction sweeps (low precision), then every request's residual.
// ev (optional, 2 events): recorded around the fused sweep launches.
int enqueue_chunk(mc_server* s, BTune g, int c, cudaStream_t st, cudaEvent_t* ev = nullptr) {
  const bool lp = s->d.dtype != MC_F64;
  const int coupled = s->d.apply == MC_APPLY_COUPLED;
  if (cudaMemcpyAsync(s->t_dev, s->t_host, sizeof(BTable), cudaMemcpyHostToDevice, st) !=
          cudaSuccess ||
      cudaMemsetAsync(s->out_dev, 0, sizeof(BOut) * kMaxReq, st) != cudaSuccess)
    return MC_ERR_CUDA;
  unsigned long long* claim = &s->t_dev->claim[0];
  if (ev && cudaEventRecord(ev[0], st) != cudaSuccess) return MC_ERR_CUDA;
  // The resident launch starts first (its clusters need whole SMs), the team and
  // queue launches run beside it (low precision: after the short b_lp_zero).  Only
  // the paths in use are launched.
  const int kind = s->d.dtype == MC_F64 ? 0 : s->d.dtype == MC_F32 ? 1 : 2;
  const int paths = table_paths(s->t_host);
  const bool queue = paths & path_bit(kPathQueue, 0);
  bool on[kSides];
  for (int i = 0; i < kSides; ++i)
    on[i] = (paths & (i < kResGroups ? path_bit(kPathResident, i)
                                     : path_bit(kPathTeam, i - kResGroups + 1))) != 0;
  auto fork = [&](cudaEvent_t e, int i0, int i1) {
    bool any = false;
    for (int i = i0; i < i1; ++i) any = any || on[i];
    if (any && cudaEventRecord(e, st) != cudaSuccess) return false;
    for (int i = i0; i < i1; ++i)
      if (on[i] && cudaStreamWaitEvent(s->side[i], e, 0) != cudaSuccess) return false;
    return true;
  };
  if (!fork(s->fork[0], 0, kResGroups)) return MC_ERR_CUDA;
  for (int i = kResGroups - 1; i >= 0; --i)   // the larger ones first
    if (on[i] && launch_resident_batch(s->t_dev, kind, coupled, i, c, s->out_dev, s->side[i]) !=
                     cudaSuccess)
      return MC_ERR_CUDA;
  if (lp && queue && b_lp_zero(s->t_dev, g, st) != cudaSuccess) return MC_ERR_CUDA;
  if (!fork(s->fork[1], kResGroups, kSides)) return MC_ERR_CUDA;
  unsigned long long* team = &s->t_dev->team_claim[0];
  cudaError_t e =
      lp ? b_lp_team(s->t_dev, team, s->out_dev, paths, kind == 2, coupled, c, s->num_sms,
                     s->side + kResGroups)
         : b_team(s->t_dev, team, s->out_dev, paths, coupled, c, s->num_sms, st,
                  s->side + kResGroups);
  if (e == cudaSuccess && queue)
    e = lp ? b_lp_sweeps(s->t_dev, claim, s->out_dev, kind == 2, coupled, c, g, st)
           : b_sweeps(s->t_dev, claim, s->out_dev, coupled, c, g, st);
  if (e != cudaSuccess) return MC_ERR_CUDA;
  for (int i = 0; i < kSides; ++i)
    if (on[i] && (cudaEventRecord(s->join[i], s->side[i]) != cudaSuccess ||
                  cudaStreamWaitEvent(st, s->join[i], 0) != cudaSuccess))
      return MC_ERR_CUDA;
  if (ev && cudaEventRecord(ev[1], st) != cudaSuccess) return MC_ERR_CUDA;
  if (lp) {
    if (b_lp_finish(s->t_dev, s->out_dev, g, st) != cudaSuccess) return MC_ERR_CUDA;
  } else {
    if (b_sweeps_finish(s->t_dev, s->out_dev, c, g, st) != cudaSuccess) return MC_ERR_CUDA;
  }
  if (b_resid(s->t_dev, s->out_dev, lp ? 1 : 0, g, st) != cudaSuccess) return MC_ERR_CUDA;
  if (cudaMemcpyAsync(s->out_host, s->out_dev, sizeof(BOut) * kMaxReq, cudaMemcpyDeviceToHost,
                      st) != cudaSuccess)
    return MC_ERR_CUDA;
  return MC_OK;
}

// Algorithmic bytes the fused sweep launches of one chunk stream: per level
// and sweep the stored operator blocks once plus the neighbour vectors read
// and the level written (FP64: 24 m^2 + 16 m inverse, 16 m^2 + 16 m coupled;
// low precision: 2 e m^2 for the two off-diagonal blocks of e-byte entries,
// + 4 m^2 for the FP32 inverse, + 16 m for the FP32 vectors d and q).
double chunk_sweep_bytes(const mc_server* s, int c) {
  const bool inv = s->d.apply == MC_APPLY_INVERSE;
  double b = 0.0;
  for (const Req* r : s->active) {
    const double m = r->chain->lay.m, L = (double)r->chain->lay.L;
    double lvl;
    if (s->d.dtype == MC_F64) {
      lvl = (inv ? 24.0 : 16.0) * m * m + 16.0 * m;
    } else {
      const double e = s->d.dtype == MC_F32 ? 4.0 : 2.0;
      lvl = 2.0 * e * m * m + (inv ? 4.0 * m * m : 0.0) + 16.0 * m;
    }
    b += lvl * L * c;
  }
  return b;
}

// Autotuner: for each batch signature (size classes present, whether any
// request is on the queue, size class of the total level count) time one live
// chunk per candidate configuration (real work, counted as such: results do not
// depend on the configuration) and keep the fastest.  Coordinate search: the persistent grid (1, 2, 3, 4,
// 6, 8 resident 256-thread blocks per SM) with one level per unit, then 2
// and 4 levels per unit, then the other bucket edge, then (low precision
// with m <= 64 present) the other load depth.
uint64_t signature(const mc_server* s) {
  const BTable* t = s->t_host;
  const int64_t lv = t->off_lv[t->n];
  int lg = 0;
  while ((1LL << lg) < lv && lg < 62) ++lg;
  uint64_t sig = (uint64_t)(lg / 2) << 8;
  for (int c = 0; c < kClasses; ++c)
    if (t->cls_end[c] > (c ? t->cls_end[c - 1] : 0)) sig |= 1ull << c;
  // the sweeps of teams and clusters do not depend on the tuned configuration: what
  // was found without a queue says nothing about one
  if (table_paths(t) & path_bit(kPathQueue, 0)) sig |= 1ull << kClasses;
  return sig;
}

// Factor status of newly admitted requests (one sync when there are any).
int check_fresh(mc_server* s) {
  bool any = false;
  for (Req* r : s->active) any |= r->fresh;
  if (!any) return MC_OK;
  if (cudaStreamSynchronize(s->user) != cudaSuccess) return MC_ERR_CUDA;
  for (size_t i = 0; i < s->active.size();) {
    Req* r = s->active[i];
    if (!r->fresh) {
      ++i;
      continue;
    }
    int32_t st = 0;
    if (cudaMemcpy(&st, &r->chain->hdr->status, sizeof(st), cudaMemcpyDeviceToHost) != cudaSuccess)
      return MC_ERR_CUDA;
    r->fresh = false;
    r->chain->factored = st == 0;
    if (st != 0) {
      retire(s, i, st, NAN, NAN, NAN, 0);
      continue;
    }
    ++i;
  }
  return MC_OK;
}

// CTAs of the launches that run side by side (deal.h).
void deal_ctas(const mc_server* s, BTable* t, const int64_t* team_levels) {
  static const int kTeams[2][kClasses] = {{8, 4, 2, 1}, {1, 2, 1, 1}};   // per CTA, by class
  const int lp = s->d.dtype != MC_F64;
  int n[kResGroups], share[kResGroups];
  for (int g = 0; g < kResGroups; ++g) {
    n[g] = t->res_end[g] - (g ? t->res_end[g - 1] : 0);
    share[g] = group_share(g);
  }
  const int cluster = resident_cluster();
  deal(DealIn{kResGroups, kClasses, n, share, team_levels, kTeams[lp], lp ? 2 : 3, s->num_sms,
              cluster > 0 ? cluster : 16, kResidentSlots},
       t->res_clusters, t->team_ctas);
}

// Whether so many FP64 requests of the resident path are active that the queue takes
// less time than the clusters, eight at a time.  By block size, requests at which the
// two took the same time for a chunk of 64 sweeps (inverse, coupled): 64 x 8 104, 105;
// 128 x 16 50, 60; 300 x 12 57; 140 x 32 25, 26; 90 x 24 23, 23; 200 x 8 none.  With
// all of them there: 250 of 128 x 16 11.0 -> 5.7 ms, 200 of 140 x 32 31.4 -> 9.6.
bool residents_overflow(const mc_server* s) {
  if (s->d.dtype != MC_F64) return false;
  double load = 0.0;
  for (const Req* r : s->active)
    if (r->path == kPathResident) {
      const int64_t m = r->chain->lay.m;
      load += m > 16 ? 1.0 / 24 : m > 8 ? 1.0 / 52 : r->chain->lay.N < 1200 ? 1.0 / 100 : 0.0;
    }
  return load > 1.0;
}

// Whether the FP64 requests of up to 16 rows on the team path run on the queue, whose
// units of several levels share a fence and a claim: from about 26000 levels together.
// A chunk of 64 sweeps by teams and by the queue, inverse: 10 of 1500 x 16 2.64, 3.19 ms,
// 6 of 3000 x 13 3.14, 3.47, 10 5.19, 5.04, 4 of 7000 x 10 4.82, 4.71, 40 of 1500 x 16
// 10.5, 9.94; coupled: 10 of 1500 x 16 1.94, 2.32, 40 7.87, 6.77.  The sums are the same.
bool small_teams_overflow(const mc_server* s) {
  int64_t levels = 0;
  for (const Req* r : s->active)
    if (r->path == kPathTeam && r->chain->lay.lp == 0 && r->chain->lay.m <= 16)
      levels += r->chain->lay.L;
  return levels >= 170ll * s->num_sms;
}

// Fill the pinned request table from the active list (small blocks first);
// returns the table order.
std::vector<Req*> build_table(mc_server* s) {
  // size classes m <= 32, 64, 128, 256, in that order
  auto cls = [](const Req* r) { return size_class(r->chain->lay.m); };
  std::stable_sort(s->active.begin(), s->active.end(),
                   [&](const Req* a, const Req* b) { return cls(a) < cls(b); });
  BTable* t = s->t_host;
  t->n = (int32_t)s->active.size();
  for (int c = 0; c < kClasses; ++c) t->cls_end[c] = 0;
  t->G = s->G;
  t->off_h1[0] = t->off_h2[0] = t->off_lv[0] = t->off_t1[0] = t->off_t2[0] = 0;
  const bool overflow = residents_overflow(s), small_queue = small_teams_overflow(s);
  // a few of the wide ones that could share an SM do not, or less, in the kernel with more
  // registers (two of 168 x 32, BF16: 0.152 -> 0.144 ms a chunk; eight of 140 x 32 two to an
  // SM 0.157, one 0.234, four 0.177)
  int wide = 0;
  for (const Req* r : s->active) wide += r->path == kPathResident && (r->group == 2 || r->group == 3);
  auto group_now = [wide](int g) {
    if (g != 2 && g != 3) return g;
    return wide <= kResidentSlots / 2 ? 4 : wide <= kResidentSlots ? 3 : g;
  };
  int64_t team_levels[kClasses] = {0, 0, 0, 0};
  const int p1 = s->d.stair == 1 ? 0 : 1;
  for (int i = 0; i < t->n; ++i) {
    const Req* r = s->active[(size_t)i];
    const int64_t L = r->chain->lay.L;
    for (int c = cls(r); c < kClasses; ++c) t->cls_end[c] = i + 1;
    fill_req(s, r, &t->r[i]);
    if (overflow && r->path == kPathResident) {
      t->r[i].path = kPathQueue;
      resident_order(r->chain->lay, &t->r[i].res_c, &t->r[i].res_s);
    }
    if (small_queue && r->path == kPathTeam && r->chain->lay.m <= 16) t->r[i].path = kPathQueue;
    const int path = t->r[i].path;
    const int64_t G = class_group(s->G, r->chain->lay.m);
    t->r[i].G = (int32_t)G;
    // units: groups of G levels of each half-sweep
    const int64_t P1 = (L - p1 + 1) / 2, P2 = (L - (1 - p1) + 1) / 2;
    const bool queue = path == kPathQueue, team = path == kPathTeam;
    t->off_h1[i + 1] = t->off_h1[i] + (queue ? (P1 + G - 1) / G : 0);
    t->off_h2[i + 1] = t->off_h2[i] + (queue ? (P2 + G - 1) / G : 0);
    t->off_t1[i + 1] = t->off_t1[i] + (team ? P1 : 0);
    t->off_t2[i + 1] = t->off_t2[i] + (team ? P2 : 0);
    t->off_lv[i + 1] = t->off_lv[i] + L;
    if (team) team_levels[cls(r)] += L;
  }
  for (int g = 0, n = 0; g < kResGroups; ++g) {
    for (int i = 0; i < t->n; ++i) {
      if (t->r[i].path == kPathResident && group_now(s->active[(size_t)i]->group) == g)
        t->res[n++] = i;
    }
    t->res_end[g] = n;
  }
  deal_ctas(s, t, team_levels);
  return std::vector<Req*>(s->active.begin(), s->active.end());
}

// After a chunk: count its sweeps and retire converged, failed and exhausted
// requests (out_host is indexed by table position).  Returns retirements.
int process_outputs(mc_server* s, const std::vector<Req*>& order, int c) {
  s->chunks++;
  int nd = 0;
  for (size_t k = 0; k < order.size(); ++k) {
    const BOut& o = s->out_host[k];
    Req* r = order[k];
    r->sweeps += c;
    // (the queue writes the epoch's counts, teams count on from their own)
    r->vbase = s->t_host->r[k].path == kPathQueue ? s->t_host->epoch + c : r->vbase + c;
    const size_t i =
        (size_t)(std::find(s->active.begin(), s->active.end(), r) - s->active.begin());
    const double kap =
        (r->step_prev > 0 && o.step > 0) ? pow(o.step / r->step_prev, 1.0 / c) : NAN;
    r->step_prev = o.step;
    if (o.status != 0) {
      retire(s, i, o.status, o.resid, o.step, kap, 0);
      ++nd;
    } else if (s->d.tol > 0 && o.resid <= s->d.tol) {
      retire(s, i, MC_OK, o.resid, o.step, kap, 1);
      ++nd;
    } else if (r->sweeps >= s->d.maxit) {
      retire(s, i, MC_ERR_NO_CONVERGENCE, o.resid, o.step, kap, 0);
      ++nd;
    }
  }
  return nd;
}

// The stream and the event of a side launch, made with its first request.
bool open_side(mc_server* s, int i) {
  return (s->side[i] || cudaStreamCreateWithFlags(&s->side[i], cudaStreamNonBlocking) == cudaSuccess) &&
         (s->join[i] ||
          cudaEventCreateWithFlags(&s->join[i], cudaEventDisableTiming) == cudaSuccess);
}

// Pinned memory, streams and events (those that exist).
void free_host_side(mc_server* s) {
  if (s->cap) cudaStreamDestroy(s->cap);
  for (cudaEvent_t f : s->fork)
    if (f) cudaEventDestroy(f);
  for (int i = 0; i < kSides; ++i) {
    if (s->side[i]) cudaStreamDestroy(s->side[i]);
    if (s->join[i]) cudaEventDestroy(s->join[i]);
  }
  if (s->t_host) cudaFreeHost(s->t_host);
  if (s->out_host) cudaFreeHost(s->out_host);
}

}  // namespace

extern "C" {

int mc_server_create(const mc_server_desc* desc, void* arena, size_t arena_bytes,
                     void* cuda_stream, mc_server** out) {
  if (!out) return MC_ERR_ARG;
  *out = nullptr;
  if (!desc || desc->check_every < 1 || desc->maxit < 1 || desc->max_active < 1 ||
      desc->max_active > kMaxReq || (desc->stair != 1 && desc->stair != 2) ||
      (desc->apply != MC_APPLY_INVERSE && desc->apply != MC_APPLY_COUPLED) ||
      (desc->dtype != MC_F64 && desc->dtype != MC_F32 && desc->dtype != MC_BF16))
    return MC_ERR_ARG;
  const size_t head = align_up(sizeof(BTable)) + align_up(sizeof(BOut) * kMaxReq);
  if (!arena || ((uintptr_t)arena & (kAlign - 1)) || arena_bytes < head + kAlign)
    return MC_ERR_WORKSPACE;
  mc_server* s = new (std::nothrow) mc_server();
  if (!s) return MC_ERR_ARG;
  s->d = *desc;
  s->arena = (char*)arena;
  s->arena_bytes = arena_bytes;
  s->user = (cudaStream_t)cuda_stream;
  s->t_dev = (BTable*)s->arena;
  s->out_dev = (BOut*)(s->arena + align_up(sizeof(BTable)));
  s->free_[head] = (arena_bytes - head) / kAlign * kAlign;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&s->num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaHostAlloc((void**)&s->t_host, sizeof(BTable), cudaHostAllocDefault) != cudaSuccess) {
    delete s;
    return MC_ERR_CUDA;
  }
  bool ok = cudaHostAlloc((void**)&s->out_host, sizeof(BOut) * kMaxReq, cudaHostAllocDefault) ==
                cudaSuccess &&
            cudaStreamCreateWithFlags(&s->cap, cudaStreamNonBlocking) == cudaSuccess &&
            cudaEventCreateWithFlags(&s->fork[0], cudaEventDisableTiming) == cudaSuccess &&
            cudaEventCreateWithFlags(&s->fork[1], cudaEventDisableTiming) == cudaSuccess;
  if (!ok) {
    free_host_side(s);
    delete s;
    return MC_ERR_CUDA;
  }
  memset(s->t_host, 0, sizeof(BTable));
  s->g_tune = BTune{2 * s->num_sms, 256, desc->dtype != MC_F64 ? 1 : 0, 0};
  s->G = 1;
  *out = s;
  return MC_OK;
}

size_t mc_server_request_bytes(const mc_server* s, int64_t L, int32_t m) {
  if (!s) return 0;
  return request_bytes(s, L, m);
}

int mc_server_submit(mc_server* s, int64_t tag, int64_t L, int32_t m, const double* dn,
                     const double* loc, const double* up) {
  if (!s || !dn || !loc || !up || L < 2 || m < 1 || m > kMaxM) return MC_ERR_ARG;
  const size_t bytes = request_bytes(s, L, m);
  if (!bytes) return MC_ERR_ARG;
  if ((int)s->active.size() >= s->d.max_active) return MC_ERR_WORKSPACE;
  size_t off = 0;
  if (!alloc(s, bytes, &off)) return MC_ERR_WORKSPACE;
  const mc_desc d = request_desc(s, L, m);
  const size_t ws = align_up(mc_workspace_bytes(&d));
  mc_chain* c = nullptr;
  int rc = chain_init(&d, s->arena + off, ws, s->user, &c);
  if (rc != MC_OK) {
    release(s, off, bytes);
    return rc;
  }
  // layout of Q^T from the host generator blocks (a row-major Q block is the
  // column-major Q^T block): T_lo[l] = up[l-1], T_up[l] = dn[l+1], T_dd = loc
  const Layout& y = c->lay;
  const size_t pe = y.plane_bytes / sizeof(double), mm = (size_t)m * m;
  const size_t dp = (size_t)y.ms * sizeof(double), sp = mm * sizeof(double);
  double* P = c->planes;
  if (cudaMemsetAsync(P + kPlaneTLO * pe, 0, dp, s->user) != cudaSuccess ||
      cudaMemcpy2DAsync(P + kPlaneTLO * pe + y.ms, dp, up, sp, sp, (size_t)(L - 1),
                        cudaMemcpyHostToDevice, s->user) != cudaSuccess ||
      cudaMemcpy2DAsync(P + kPlaneTUP * pe, dp, dn + mm, sp, sp, (size_t)(L - 1),
                        cudaMemcpyHostToDevice, s->user) != cudaSuccess ||
      cudaMemsetAsync(P + kPlaneTUP * pe + (size_t)(L - 1) * y.ms, 0, dp, s->user) !=
          cudaSuccess ||
      cudaMemcpy2DAsync(P + kPlaneTDD * pe, dp, loc, sp, sp, (size_t)L, cudaMemcpyHostToDevice,
                        s->user) != cudaSuccess)
    rc = MC_ERR_CUDA;
  if (rc == MC_OK &&
      cudaMemsetAsync(c->fver, 0, (size_t)L * sizeof(int), s->user) != cudaSuccess)
    rc = MC_ERR_CUDA;
  if (rc == MC_OK && launch_block_exp(P, chain_bexp(c, 0), y, s->user) != cudaSuccess)
    rc = MC_ERR_CUDA;
  if (rc == MC_OK) rc = chain_factor_async(c);
  if (rc == MC_OK && launch_fill(c->xa, y.N, 1.0 / (double)y.N, s->user) != cudaSuccess)
    rc = MC_ERR_CUDA;
  if (rc == MC_OK && y.lp) rc = chain_residual_async(c, c->xa, s->user, chain_lpQ(c));
  if (rc != MC_OK) {
    mc_destroy(c);
    release(s, off, bytes);
    return rc;
  }
  Req* r = new (std::nothrow) Req();
  if (!r) {
    mc_destroy(c);
    release(s, off, bytes);
    return MC_ERR_ARG;
  }
  r->tag = tag;
  r->chain = c;
  r->off = off;
  r->bytes = bytes;
  r->lsum = (double*)(s->arena + off + ws);
  r->sweeps = 0;
  r->step_prev = NAN;
  r->path = b_path(y, s->d.apply == MC_APPLY_COUPLED, s->num_sms);
  r->group = resident_batch_group(y, s->d.apply == MC_APPLY_COUPLED);
  const int side = r->path == kPathResident ? r->group
                   : r->path == kPathTeam   ? kResGroups - 1 + size_class(m)
                                            : -1;
  bool ok = side < (r->path == kPathTeam ? kResGroups : 0) || open_side(s, side);
  if (side == 2 || side == 3) ok = ok && open_side(s, 3) && open_side(s, 4);   // build_table
  // a chain that would stay on chip by itself has no row exponents yet; teams use them
  if (ok && c->res_ctas && y.lp == 0 && m > 16 && r->path == kPathTeam)
    ok = launch_weak_rows(P, chain_bexp(c, 0), y, s->d.apply == MC_APPLY_COUPLED, s->user) ==
         cudaSuccess;
  if (!ok) {
    mc_destroy(c);
    release(s, off, bytes);
    delete r;
    return MC_ERR_CUDA;
  }
  r->vbase = 0;
  r->fresh = true;
  if (reset_team_words(s, r) != cudaSuccess) {
    mc_destroy(c);
    release(s, off, bytes);
    delete r;
    return MC_ERR_CUDA;
  }
  s->active.push_back(r);
  return MC_OK;
}

int mc_server_step(mc_server* s, int32_t* n_active, int32_t* n_done) {
  if (!s) return MC_ERR_ARG;
  const int c = s->d.check_every;
  int rc = check_fresh(s);
  if (rc != MC_OK) return rc;
  if (!s->active.empty()) {
    const bool lp = s->d.dtype != MC_F64;
    s->G = 1;
    std::vector<Req*> order = build_table(s);
    const uint64_t sig = signature(s);
    auto it = s->tuned.find(sig);
    if (it == s->tuned.end() && s->d.autotune) {
      // candidate list: grids first (G = 1, default edges and depth), then
      // the other knobs around the best so far
      const BTune base{2 * s->num_sms, 256, lp ? 1 : 0, 0};
      BTune best = base;
      int bestG = 1;
      float best_ms = 1e30f;
      cudaEvent_t ev[4] = {nullptr, nullptr, nullptr, nullptr};
      for (cudaEvent_t& e : ev)
        if (cudaEventCreate(&e) != cudaSuccess) return MC_ERR_CUDA;
      const bool small_lp = lp && (sig & 3ull) != 0;
      static const int kGrid[] = {1, 2, 3, 4, 6, 8};
      bool stop = false;
      for (int stage = 0; stage < 4 && !stop && rc == MC_OK; ++stage) {
        const int ncand = stage == 0 ? 6 : stage == 1 ? 2 : (stage == 3 && !small_lp) ? 0 : 1;
        for (int ci = 0; ci < ncand && !stop && rc == MC_OK; ++ci) {
          BTune g = best;
          int G = bestG;
          if (stage == 0) g.blocks = kGrid[ci] * s->num_sms;
          if (stage == 1) G = ci == 0 ? 2 : 4;
          if (stage == 2) g.split64 = 1 - best.split64;
          if (stage == 3) g.deep = 1 - best.deep;
          s->G = G;
          order = build_table(s);
          if (cudaEventRecord(ev[0], s->user) != cudaSuccess) rc = MC_ERR_CUDA;
          if (rc == MC_OK) rc = begin_chunk(s, c);
          if (rc == MC_OK) rc = enqueue_chunk(s, g, c, s->user, ev + 1);
          if (rc == MC_OK && cudaEventRecord(ev[3], s->user) != cudaSuccess) rc = MC_ERR_CUDA;
          if (rc == MC_OK && cudaEventSynchronize(ev[3]) != cudaSuccess) rc = MC_ERR_CUDA;
          float ms = 0.0f, sw = 0.0f;
          if (rc == MC_OK && (cudaEventElapsedTime(&ms, ev[0], ev[3]) != cudaSuccess ||
                              cudaEventElapsedTime(&sw, ev[1], ev[2]) != cudaSuccess))
            rc = MC_ERR_CUDA;
          if (rc != MC_OK) break;
          mc_server_tuning tr{};
          tr.signature = sig;
          tr.blocks_per_sm = g.blocks / s->num_sms;
          tr.levels_per_unit = G;
          tr.split64 = g.split64;
          tr.deep = g.deep;
          tr.chunk_ms = ms;
          tr.sweep_ms = sw;
          tr.sweep_bytes = chunk_sweep_bytes(s, c);
          s->trials.push_back(tr);
          if (ms < best_ms) {
            best_ms = ms;
            best = g;
            bestG = G;
          }
          stop = process_outputs(s, order, c) > 0 || s->active.empty();
        }
      }
      for (cudaEvent_t e : ev) cudaEventDestroy(e);
      if (rc != MC_OK) return rc;
      s->tuned[sig] = best;
      s->tuned_G[sig] = bestG;
      for (mc_server_tuning& tr : s->trials)
        if (tr.signature == sig)
          tr.chosen = tr.blocks_per_sm == best.blocks / s->num_sms && tr.levels_per_unit == bestG &&
                      tr.split64 == best.split64 && tr.deep == best.deep;
    } else {
      BTune g{2 * s->num_sms, 256, lp ? 1 : 0, 0};
      int G = 1;
      if (it != s->tuned.end()) {
        g = it->second;
        G = s->tuned_G[sig];
      }
      if (G != s->G) {
        s->G = G;
        order = build_table(s);
      }
      const int paths = table_paths(s->t_host);
      if (!s->gexec || s->g_chunk != c || s->g_paths != paths || s->g_tune.blocks != g.blocks ||
          s->g_tune.threads != g.threads || s->g_tune.split64 != g.split64 ||
          s->g_tune.deep != g.deep) {
        if (s->gexec) {
          cudaGraphExecDestroy(s->gexec);
          s->gexec = nullptr;
        }
        if (cudaStreamBeginCapture(s->cap, cudaStreamCaptureModeThreadLocal) != cudaSuccess)
          return MC_ERR_CUDA;
        rc = enqueue_chunk(s, g, c, s->cap);
        cudaGraph_t gr = nullptr;
        const cudaError_t e = cudaStreamEndCapture(s->cap, &gr);
        if (rc != MC_OK || e != cudaSuccess) {
          if (gr) cudaGraphDestroy(gr);
          cudaGetLastError();
          return MC_ERR_CUDA;
        }
        const cudaError_t e2 = cudaGraphInstantiate(&s->gexec, gr, 0);
        cudaGraphDestroy(gr);
        if (e2 != cudaSuccess) {
          s->gexec = nullptr;
          return MC_ERR_CUDA;
        }
        s->g_chunk = c;
        s->g_paths = paths;
        s->g_tune = g;
      }
      rc = begin_chunk(s, c);
      if (rc != MC_OK) return rc;
      if (cudaGraphLaunch(s->gexec, s->user) != cudaSuccess ||
          cudaStreamSynchronize(s->user) != cudaSuccess)
        return MC_ERR_CUDA;
      process_outputs(s, order, c);
    }
  }
  if (n_active) *n_active = (int32_t)s->active.size();
  if (n_done) *n_done = (int32_t)s->done.size();
  return MC_OK;
}

int mc_server_fetch(mc_server* s, int64_t* tag, double* pi_host, int64_t n_cap, mc_result* res,
                    int32_t* status) {
  if (!s || s->done.empty()) return MC_ERR_ARG;
  Done dn = s->done.front();
  if (pi_host && n_cap < dn.N) return MC_ERR_ARG;
  s->done.pop_front();
  if (tag) *tag = dn.tag;
  if (pi_host && dn.pi) memcpy(pi_host, dn.pi, sizeof(double) * (size_t)dn.N);
  if (res) *res = dn.res;
  if (status) *status = dn.status;
  free(dn.pi);
  return MC_OK;
}

int mc_server_grid(const mc_server* s, int32_t* blocks, int32_t* threads, int32_t* n_tuned) {
  if (!s) return MC_ERR_ARG;
  if (blocks) *blocks = s->g_tune.blocks;
  if (threads) *threads = s->g_tune.threads;
  if (n_tuned) *n_tuned = (int32_t)s->tuned.size();
  return MC_OK;
}

int mc_server_trials(const mc_server* s, mc_server_tuning* out, int32_t cap, int32_t* n) {
  if (!s || cap < 0 || (cap > 0 && !out)) return MC_ERR_ARG;
  const int32_t total = (int32_t)s->trials.size();
  for (int32_t i = 0; i < total && i < cap; ++i) out[i] = s->trials[(size_t)i];
  if (n) *n = total;
  return MC_OK;
}

void mc_server_destroy(mc_server* s) {
  if (!s) return;
  cudaStreamSynchronize(s->user);
  while (!s->active.empty()) {
    Req* r = s->active.back();
    mc_destroy(r->chain);
    delete r;
    s->active.pop_back();
  }
  for (Done& dn : s->done) free(dn.pi);
  if (s->gexec) cudaGraphExecDestroy(s->gexec);
  free_host_side(s);
  delete s;
}

}  // extern "C"
