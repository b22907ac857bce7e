// Instantiations of pe_eval_slot_kernel: plain.
#include "pe_slot_launch.h"

namespace pe {
int launch_slot_plain(const SlotCall& t) { return launch_slot_mode<kSlotPlain>(t); }
}  // namespace pe
