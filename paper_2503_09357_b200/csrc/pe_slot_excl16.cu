// Instantiations of pe_eval_slot_kernel: exclusive channels, 16-bit channel words.
#include "pe_slot_launch.h"

namespace pe {
int launch_slot_excl16(const SlotCall& t) { return launch_slot_mode<kSlotExcl16>(t); }
}  // namespace pe
