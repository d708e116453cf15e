// How a chunk's launches share the GPU (plain C++: also compiled by a CPU test).
//
// Clusters take `cluster` SMs whole, a slot that share[g] clusters of a group g can use
// at the same time.  Slots go one by one to the group with the most requests in turn,
// half of `most_slots` where teams run too; every group with requests has one.  The
// teams share the other SMs, per_sm CTAs each, in proportion to their levels, so that
// each gets its part at once instead of the first launch filling the GPU for a
// chunk's time: no more than one team per level, at least one CTA per class that
// has levels.  No result depends on it.
#pragma once
#include <stdint.h>

namespace mc {

struct DealIn {
  int groups, classes;
  const int* n;               // requests per group
  const int* share;
  const int64_t* team_levels; // levels per class
  const int* teams_per_cta;
  int per_sm, sms, cluster, most_slots;
};

inline void deal(const DealIn& d, int32_t* clusters, int32_t* team_ctas) {
  int64_t want[8] = {}, sum = 0;
  for (int c = 0; c < d.classes; ++c) {
    want[c] = (d.team_levels[c] + d.teams_per_cta[c] - 1) / d.teams_per_cta[c];
    sum += want[c];
  }
  int slots[8] = {}, used = 0, present = 0;
  for (int g = 0; g < d.groups; ++g) present += d.n[g] > 0;
  int left = sum > 0 ? d.most_slots / 2 : d.most_slots;
  if (left > d.sms / d.cluster) left = d.sms / d.cluster;
  if (left < present) left = present;
  for (; left > 0; --left) {
    int best = -1;
    double turns = 1.0;   // requests per cluster: no group needs more clusters than requests
    for (int g = 0; g < d.groups; ++g) {
      const double r = d.n[g] == 0  ? 0.0
                       : slots[g] ? (double)d.n[g] / (slots[g] * d.share[g])
                                  : 2e9;
      if (r > turns) best = g, turns = r;
    }
    if (best < 0) break;
    ++slots[best];
    ++used;
  }
  for (int g = 0; g < d.groups; ++g) {
    const int most = slots[g] * d.share[g];
    clusters[g] = d.n[g] < most ? d.n[g] : most;
  }
  int64_t free_ctas = (int64_t)d.per_sm * (d.sms - d.cluster * used);
  if (free_ctas < 1) free_ctas = 1;
  for (int c = 0; c < d.classes; ++c) {
    int64_t n = want[c];
    if (sum > free_ctas) n = (n * free_ctas + sum - 1) / sum;   // >= 1 where want >= 1
    team_ctas[c] = (int32_t)n;
  }
}

}  // namespace mc
