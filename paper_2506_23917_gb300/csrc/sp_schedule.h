// sp_schedule.h -- the collision schedules the autotuner tries (host only).
#pragma once
#include <algorithm>
#include <utility>
#include <vector>

namespace sp {

// (cap, warps): for each block size the fixed capacities, and the largest
// capacity at each residency level (blocks per SM from the occupancy
// calculator): more resident warps with slightly smaller batches can win (on
// the developed cylinder 864 x 2 at 6 blocks beat 1024 x 2 at 5 by 2 %).
// fits(cap, warps): whether sp_set_schedule takes it; blocks(cap, warps):
// resident blocks per SM.  A capacity that is refused stands for no level:
// the largest one below it that is taken does.
template <class Fits, class Blocks>
std::vector<std::pair<int, int>> schedule_candidates(int cap_max, Fits fits, Blocks blocks) {
  std::vector<std::pair<int, int>> out;
  const auto add = [&](int cap, int warps) {
    const auto s = std::make_pair(cap, warps);
    if (std::find(out.begin(), out.end(), s) == out.end()) out.push_back(s);
  };
  for (int warps : {2, 4, 8}) {
    for (int cap : {128, 256, 384, 512, 768, 1024})
      if (fits(cap, warps)) add(cap, warps);
    int last = -1;
    for (int cap = cap_max; cap >= 128; cap -= 32) {
      if (!fits(cap, warps)) continue;
      const int per = blocks(cap, warps);
      if (per != last && per > 0) add(cap, warps);
      last = per;
    }
  }
  return out;
}

}  // namespace sp
