// Internal: shape of a pe_eval_tile_kernel launch (computed by plan_tile, read by the kernel).
#pragma once
#include <stdint.h>

namespace pe {

constexpr int kTileWarps = 8;   // warps of a block (twice as many where operators are few)

// MODE of the kernel (Plan::tile_mode)
constexpr int kTilePlain = 0;   // 32-bit state words
constexpr int kTileS16 = 1;     // 16-bit state words
constexpr int kTileExcl = 2;    // PE_COMM_EXCLUSIVE: the end of the last transfer per channel, [machine pair][P]
constexpr int kTileHet = 3;     // durations by machine
constexpr int kTileLong = 4;    // 32-bit state words, time bounds up to kPackedTimeLimit
constexpr int kTileExclLong = 5;

struct TileShape {
  int lanes;            // P, candidates per tile (4 to 32)
  int jbits;            // machine bits of a state word (8 with 32-bit words)
  int64_t tiles;        // ceil(K / P)
  uint32_t off_dev;     // byte offsets in shared memory: machine records of warp 0, weight sums, state words, channels
  uint32_t off_wsum;
  uint32_t off_state;
  uint32_t off_chan;
  uint32_t dev_bytes;   // bytes per warp of each area (state: per pair of warps with 16-bit words)
  uint32_t wsum_bytes;
  uint32_t state_bytes;
  uint32_t chan_bytes;
  int vector_init;      // assignments can be read four candidates at a time
};

}  // namespace pe
