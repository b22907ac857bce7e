// pe_eval_tile_kernel: instantiations of one assignment layout and mode.
#include "pe_tile_launch.h"

namespace pe {

int launch_tile_op_excl(const TileCall& t) { return launch_tile_mode<false, kTileExcl>(t); }

}  // namespace pe
