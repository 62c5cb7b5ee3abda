// Host-side choice of the work items per tile of an FP64 stage launch.
#pragma once
#include <algorithm>
#include <map>
#include <vector>

namespace rlb {

constexpr int SPLIT_MAX = 8;  // most work items per tile

// Consecutive tiles of a launch with equally many velocity rows.
struct TileRun {
  double rows;
  long long tiles;
};

// Work items per tile of the FP64 stage kernel. The velocity rows of a tile are split over several CTAs where that
// shortens the launch: for each split the tiles, in their order, are handed to `slots` resident CTAs as they come
// free, an item costing its rows plus a fixed part worth ROW0 rows (the per-cell chain, barriers and start-up: 12 to 16
// us on GB300, where a CTA takes 0.6 us per row), and the split with the earliest end is taken. Handles of
// many times the slots are never split. Against "split only what cannot fill the slots": 13 uneven tubes, 545
// tiles of 16 to 288 rows for 456 slots, 137 -> 115 us per stage.
//
// Slots that come free at the same time are held together, and a larger split is looked at only while the work
// spread evenly over the slots (which grows with the split) could still end earlier: equal tiles take one step per
// wave instead of one per item. 3647 equal tiles: under 1 us on one x86 core, 3.1 ms with a queue of single slots; 500
// tubes of 7 tiles: 0.06 and 9.9 ms.
inline int choose_split(const std::vector<TileRun>& runs, long long slots) {
  constexpr double ROW0 = 20;
  long long n = 0;
  double rows = 0.0;
  for (const TileRun& r : runs) {
    n += r.tiles;
    rows += r.rows * (double)r.tiles;
  }
  if (n >= 8 * slots) return 1;
  int best = 1;
  double best_end = -1.0;
  for (int s = 1; s <= SPLIT_MAX; ++s) {
    if (best_end >= 0.0 && (ROW0 * (double)(n * s) + rows) / (double)slots >= best_end) break;
    std::map<double, long long> free_at;  // time -> slots that come free then
    free_at[0.0] = slots;
    double end = 0.0;
    for (const TileRun& r : runs) {
      const double cost = ROW0 + r.rows / s;
      for (long long left = r.tiles * s; left > 0;) {
        const auto first = free_at.begin();
        const long long k = std::min(first->second, left);
        const double at = first->first + cost;
        if ((first->second -= k) == 0) free_at.erase(first);
        free_at[at] += k;
        end = std::max(end, at);
        left -= k;
      }
    }
    if (best_end < 0.0 || end < best_end) {
      best_end = end;
      best = s;
    }
  }
  return best;
}

}  // namespace rlb
