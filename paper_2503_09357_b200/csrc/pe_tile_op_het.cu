// pe_eval_tile_kernel: instantiations of one assignment layout and mode.
#include "pe_tile_launch.h"

namespace pe {

int launch_tile_op_het(const TileCall& t) { return launch_tile_mode<false, kTileHet>(t); }

}  // namespace pe
