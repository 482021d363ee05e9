// heom_team.h -- the team size (CTAs per hierarchy) of a batch launch.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <functional>
#include <queue>
#include <vector>

namespace heom {

constexpr int kTeamSizes[5] = {1, 2, 4, 8, 16};

// Of 1, 2, 4, 8 and 16 CTAs the size whose longest-first packing of hierarchies of `blocks` node blocks onto the teams
// that the GPU holds at once has the shortest makespan, with a stage of b node blocks per CTA taking 1.5 + m b us, 1.2
// + m b where the team is one CTA, which has no cluster barrier (measured: 1.0 for a block, and a little more where its
// sets' last round is partly filled).  us per step, mixed: 3 sites of 2 to 6 blocks 4.4 to 5.6 against 7.1 to 7.4 in a
// cluster, 4 sites of 2 and 3 blocks 4.5 and 5.1 against 7.2 (of 7 blocks 8.3 against 7.4: a cluster is picked).
// resident[i]: teams of kTeamSizes[i] CTAs that the GPU holds at once; 0: none, the size is not considered.  (A cluster
// does not span the GPU's processing clusters, so fewer teams fit than SMs / size: 76, 36, 15 and 7 of 2, 4, 8 and 16
// CTAs on 152 SMs.)
inline int pick_team(std::vector<int64_t> blocks, double m, const int* resident) {
  std::sort(blocks.begin(), blocks.end(), std::greater<int64_t>());
  int best = 1;
  double best_t = -1.0;
  for (int i = 0; i < 5; ++i) {
    if (resident[i] < 1) continue;
    const int c = kTeamSizes[i];
    std::priority_queue<double, std::vector<double>, std::greater<double>> load;
    for (size_t t = 0; t < std::min<size_t>(blocks.size(), resident[i]); ++t) load.push(0.0);
    double span = 0.0;
    for (int64_t b : blocks) {
      const double t = load.top() + (c == 1 ? 1.2 : 1.5) + m * (double)((b + c - 1) / c);
      load.pop();
      load.push(t);
      span = std::max(span, t);
    }
    if (best_t < 0.0 || span < 0.98 * best_t) {
      best = c;
      best_t = span;
    }
  }
  return best;
}

}  // namespace heom
