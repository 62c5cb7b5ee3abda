// Test-only shim: the library's choice of the split (csrc/rlb_schedule.h) beside the same rule with a queue of single
// slots, and the time each takes. Built by tests/test_schedule_cpu.py; not part of the library.
#include <chrono>
#include <functional>
#include <queue>

#include "../../paper_1608_03004_gb300/csrc/rlb_schedule.h"

static int single_slots(const std::vector<rlb::TileRun>& runs, long long slots) {
  long long n = 0;
  for (const auto& r : runs) n += r.tiles;
  if (n >= 8 * slots) return 1;
  int best = 1;
  double best_end = -1.0;
  for (int s = 1; s <= rlb::SPLIT_MAX; ++s) {
    std::priority_queue<double, std::vector<double>, std::greater<double>> free_at;
    double end = 0.0;
    for (const auto& r : runs)
      for (long long k = 0; k < r.tiles * s; ++k) {
        double at = 0.0;
        if ((long long)free_at.size() >= slots) {
          at = free_at.top();
          free_at.pop();
        }
        at += 20 + r.rows / s;
        end = std::max(end, at);
        free_at.push(at);
      }
    if (best_end < 0.0 || end < best_end) {
      best_end = end;
      best = s;
    }
  }
  return best;
}

// out[0], out[1]: the library's choice and the rule's; us[0], us[1]: their shortest times of three.
extern "C" void schedule_eval(const double* rows, const long long* tiles, int n, long long slots, int* out, double* us) {
  std::vector<rlb::TileRun> runs;
  for (int k = 0; k < n; ++k) runs.push_back({rows[k], tiles[k]});
  for (int w = 0; w < 2; ++w)
    for (int rep = 0; rep < 3; ++rep) {
      const auto t0 = std::chrono::steady_clock::now();
      out[w] = w == 0 ? rlb::choose_split(runs, slots) : single_slots(runs, slots);
      const double t = std::chrono::duration<double, std::micro>(std::chrono::steady_clock::now() - t0).count();
      us[w] = rep == 0 ? t : std::min(us[w], t);
    }
}
