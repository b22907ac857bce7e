// pe_eval_tile_kernel: instantiations of one assignment layout, time bounds beyond 2^23, with and without channels.
#include "pe_tile_launch.h"

namespace pe {

int launch_tile_pos_long(const TileCall& t) {
  return t.p->tile_mode == kTileExclLong ? launch_tile_mode<true, kTileExclLong>(t) : launch_tile_mode<true, kTileLong>(t);
}

}  // namespace pe
