// Instantiations of pe_eval_slot_kernel: durations by machine.
#include "pe_slot_launch.h"

namespace pe {
int launch_slot_het(const SlotCall& t) { return launch_slot_mode<kSlotHet>(t); }
}  // namespace pe
