// Internal: shape of a pe_eval_slot_kernel launch (computed by plan_slot, read by the kernel).
#pragma once
#include <stdint.h>

namespace pe {

constexpr int kSlotWarps = 16;   // most warps of a block
constexpr int kSlotQuads = 2;    // groups of four positions that are requested together

struct SlotShape {
  int lanes;            // P, candidates per tile
  int64_t tiles;        // ceil(candidates of the chunk / P)
  uint32_t off_ring;    // byte offsets in shared memory: requested words of warp 0, machine records, channel words, slots
  uint32_t off_dev;
  uint32_t off_chan;
  uint32_t off_state;
  uint32_t dev_bytes;   // bytes per warp of each area
  uint32_t chan_bytes;
  uint32_t state_bytes;
};

}  // namespace pe
