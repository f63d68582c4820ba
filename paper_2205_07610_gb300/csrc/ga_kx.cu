// ga_kx.cu -- choice of the strip tile (ga_kx.h).
#include "ga_kx.h"

#include <algorithm>

namespace ga {

namespace {
struct Step {  // cycles per row of a scheduler: max(lone, warps * each + fixed)
  int lone, each, fixed;
};
// Without a profile, local and global mode / semi-global mode; with one, the same.
// Columns: kKx4, kKx8, kKx12, kKx16, kKx20, kKx8Wide, kKx16Wide (0: no such kernel).
constexpr Step kSteps[4][kKxTiles] = {
    {{94, 57, 0}, {115, 93, 0}, {155, 137, 0}, {220, 181, 0}, {265, 224, 0}, {}, {290, 145, 60}},
    {{104, 52, 0}, {172, 84, 40}, {230, 105, 50}, {}, {}, {}, {290, 160, 60}},
    {{95, 66, 0}, {150, 114, 0}, {}, {}, {}, {175, 103, 20}, {}},
    {{104, 66, 0}, {175, 103, 20}, {}, {}, {}, {}, {}}};
}  // namespace

int kx_choose(int mode, bool profile, const int64_t *chain, const int64_t *strips, int nsm, double *cycles) {
  const Step *tab = kSteps[(profile ? 2 : 0) + (mode == 2 ? 1 : 0)];
  const int64_t sched = 4 * (int64_t)nsm;
  int best = -1;
  double tbest = 0;
  for (int i = 0; i < kKxTiles; ++i) {
    if (!tab[i].lone) continue;
    const int64_t n = strips[kKxTileK[i] / 4 - 1], w = (n + sched - 1) / sched;
    const double step = std::max<double>(tab[i].lone, (double)(w * tab[i].each + tab[i].fixed));
    const double t = (double)chain[kKxTileK[i] / 4 - 1] * step;
    if (best < 0 || t < tbest) {
      best = i;
      tbest = t;
    }
  }
  if (cycles) *cycles = tbest;
  return best;
}

}  // namespace ga
