// Variant and pipeline rings of the fp32 tensor-core kernel (umma_conv_f32.cu) for a bundle width.  Host only.
#pragma once

#include <cstddef>

namespace rt3d {

constexpr int kSplitSlots = 4;                          // most A operands in tensor memory
constexpr int kSplitInputs = 8;                         // most staged inputs
constexpr int kSplitSlotCols = 48;                      // tensor-memory columns of one: three parts of 32 channels, two to a column
constexpr int kSplitInputBytes = 128 * 128;             // 128 voxels x 32 fp32 channels
constexpr int kSplitDrainStage = 32 * 64;               // bytes with which a drain warp turns 32 voxels x 16 channels
constexpr int kSplitBarBytes = 344;                     // the kernel's barriers
constexpr size_t kSplitSmem = 227 * 1024;

// Where the accumulators of the small products lie (umma_conv_f32.cu).
enum SplitMode { kSplitNone, kSplitSmall, kSplitAll };

// Columns that a drain thread holds, steps per hand-shake, how the accumulators lie, CTA pairs.
// Up to 64 columns single CTAs win with three or four MMAs a slice, above that pairs do: half of the weights' traffic in shared
// memory, and the MMAs are as wide as they take to issue.  64 -> 128 channels 3x3x3 on 2 x 16 x 56 x 56: pairs 168 us, single
// CTAs 192; 88 -> 41 on 2 x 14 x 59 x 12: 65 and 56.  Two steps per hand-shake where tensor memory holds two such A operands
// (64 -> 32 on 2 x 16 x 56 x 56 149 -> 117 us).
struct SplitVariant { int nh, sub; SplitMode mode; bool pair; };
inline SplitVariant split_variant(int n_tile) {
  if (n_tile <= 32) return {16, 2, kSplitAll, false};
  if (n_tile <= 48) return {32, 2, kSplitAll, false};
  if (n_tile <= 64) return {32, 2, kSplitSmall, false};
  if (n_tile <= 96) return {48, 2, kSplitNone, true};
  return {64, 1, kSplitNone, true};
}

// Staged inputs, weight stages and A operands of a CTA, in hand-shakes.
struct SplitRing { int inputs, stages, slots; };

inline size_t split_smem_bytes(int n_tile, int n_bundles, const SplitRing& r) {
  const SplitVariant v = split_variant(n_tile);
  return 1024 + size_t(v.sub) * (size_t(r.inputs) * kSplitInputBytes + size_t(r.stages) * n_tile * (v.pair ? 96 : 192)) +
         8 * kSplitDrainStage + kSplitBarBytes + 16 + size_t(n_tile) * n_bundles * 4;
}

// Whether the two splitting teams, which take the staged inputs in turn, find every input complete that they wait for.  A wait
// on a barrier's phase is answered by the completion before the last as well, so a team may only wait for a buffer whose last
// fill it knows to have landed.  With an even number of buffers it has waited for that fill itself; with an odd one the other
// team has, and what orders it is the MMAs of slots + 2 hand-shakes ago, which this team has waited for.
inline bool split_inputs_ordered(const SplitRing& r) { return r.inputs % 2 == 0 || r.inputs >= r.slots + 2; }

// False where shared memory does not hold a pipeline.  A weight stage more than A operands in flight is the least (the MMAs of a
// slot's last operand free its weights later than the slot); two more are taken where four inputs fit beside them.
inline bool split_ring(int n_tile, int n_bundles, SplitRing* out) {
  if (n_tile % 16 || n_tile < 16 || n_tile > 128 || n_bundles < 1) return false;
  const SplitVariant v = split_variant(n_tile);
  const int acc = (v.mode == kSplitAll ? 6 : v.mode == kSplitSmall ? 4 : 3) * n_tile, room = (512 - acc) / (v.sub * kSplitSlotCols);
  SplitRing r;
  r.slots = room < kSplitSlots ? room : kSplitSlots;
  for (int fewest = 4; fewest >= 2; fewest -= 2)
    for (r.stages = r.slots + 2; r.stages > r.slots; --r.stages)
      for (r.inputs = kSplitInputs; r.inputs >= fewest; --r.inputs)
        if (split_inputs_ordered(r) && split_smem_bytes(n_tile, n_bundles, r) <= kSplitSmem) {
          *out = r;
          return true;
        }
  return false;
}

}  // namespace rt3d
