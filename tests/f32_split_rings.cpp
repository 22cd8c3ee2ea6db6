// The pipeline rings of the fp32 tensor-core kernel, walked hand-shake by hand-shake for every bundle width and for as many
// bundles as shared memory takes (their biases shrink the rings): when a role waits for a fill of a buffer, the fill before it
// must be known to have landed, because a parity wait is answered by that one's predecessor as well.  Built with the header alone.
#include <cstdio>
#include <set>

#include "f32_split_plan.h"

using namespace rt3d;

int main() {
  int plans = 0;
  std::set<int> seen;
  for (int n_tile = 16; n_tile <= 128; n_tile += 16)
    for (int bundles = 1;; ++bundles) {
      SplitRing r;
      if (!split_ring(n_tile, bundles, &r)) {
        if (bundles * n_tile < 2048) { std::printf("no plan: %d x %d\n", n_tile, bundles); return 1; }
        break;
      }
      ++plans;
      if (split_smem_bytes(n_tile, bundles, r) > kSplitSmem || r.inputs > kSplitInputs || r.slots < 2 || r.slots > kSplitSlots ||
          r.stages <= r.slots || r.stages > 8)
        return std::printf("limits: %d x %d: %d %d %d\n", n_tile, bundles, r.inputs, r.stages, r.slots), 1;
      if (!seen.insert(((n_tile * 16 + r.inputs) * 16 + r.stages) * 16 + r.slots).second) continue;
      std::printf("%d columns from %d bundles: %d inputs, %d stages, %d slots\n", n_tile, bundles, r.inputs, r.stages, r.slots);
      // what each team knows: the latest hand-shake whose MMAs it has waited for, and the inputs that it has waited for itself
      int mma_done[2] = {-1, -1};
      std::set<int> landed[2];
      for (int c = 0; c < 1000; ++c) {
        const int team = c & 1;
        const int in = c - r.inputs, w = c - r.stages, e = c - r.slots - r.stages;
        // x_full: the input of hand-shake c, before any other wait of this turn
        if (in >= 0 && !landed[team].count(in) && in > mma_done[team])
          return std::printf("%d x %d: the input of hand-shake %d is waited for while that of %d may be on its way\n", n_tile, bundles, c, in), 1;
        landed[team].insert(c);
        // empty: the MMAs of hand-shake c - slots, whose stage was used by c - slots - stages before
        if (e >= 0 && e > mma_done[team]) return std::printf("%d x %d: slot of hand-shake %d\n", n_tile, bundles, c), 1;
        if (c >= r.slots) mma_done[team] = c - r.slots;
        // full (pairs): the weights of hand-shake c
        if (w >= 0 && w > mma_done[team]) return std::printf("%d x %d: weights of hand-shake %d\n", n_tile, bundles, c), 1;
      }
    }
  SplitRing odd = {3, 4, 2}, odd16 = {5, 6, 4}, far = {5, 5, 3};
  if (split_inputs_ordered(odd) || split_inputs_ordered(odd16) || !split_inputs_ordered(far)) return std::printf("rule\n"), 1;
  std::printf("%d plans\nok\n", plans);
  return 0;
}
