// Internal: launch templates of pe_eval_slot_kernel.  The instantiations are spread over one translation unit per kernel
// mode (pe_slot_*.cu) so that they compile in parallel.
#pragma once
#include "pe_kernel_slot.cuh"
#include "pe_launch.h"

namespace pe {

// One chunk of a batch: outputs start at its first candidate, entries, status, wsum and words are in the workspace.
struct SlotCall {
  const pe_graph* g;
  const Plan* p;
  int64_t K;         // row pitch of the interface arrays
  int64_t n;         // candidates of the chunk
  int64_t pitch;     // row pitch of the workspace arrays
  const uint4* entries;
  const uint32_t* status;
  const int32_t* wsum;
  uint32_t* words;   // times by operator
  SlotShape shape;
  int64_t grid;
  pe_outputs out;
  cudaStream_t stream;
};

template <int CLS, int EDGES, int MODE, bool OWN = false>
int launch_slot3(const SlotCall& t) {
  auto go = [&](auto kern) -> int {
    if (!set_smem(kern, t.p->smem)) return PE_ERR_CUDA;
    kern<<<(unsigned)t.grid, t.p->threads, t.p->smem, t.stream>>>(t.g->sview, t.g->d_sblob, t.K, t.n, t.entries, t.pitch, t.status,
                                                                 t.wsum, t.words, t.out, t.g->d_error, t.shape);
    return PE_OK;
  };
  if (!t.out.start) return go(pe_eval_slot_kernel<CLS, EDGES, 0, MODE, OWN>);
  if (t.words) return go(pe_eval_slot_kernel<CLS, EDGES, 2, MODE, OWN>);
  return go(pe_eval_slot_kernel<CLS, EDGES, 1, MODE, OWN>);
}

template <int MODE>
int launch_slot_mode(const SlotCall& t) {
  const PeSlotView& v = t.g->sview;
  constexpr bool kPlain = MODE == kSlotPlain, kExcl = MODE == kSlotExcl || MODE == kSlotExcl16;
  if constexpr (!kExcl) {
    if (v.marks) {
      if (v.max_sources <= 1) return launch_slot3<0, 1, MODE, true>(t);
      if (v.max_sources == 2) return launch_slot3<0, 2, MODE, true>(t);
      return launch_slot3<0, 3, MODE, true>(t);
    }
  } else if (v.marks) {
    return PE_ERR_UNSUPPORTED;
  }
  const bool eight = v.max_sources <= 8;
  if (v.cls_kind == 0) {
    if (kPlain && v.max_sources <= 1) return launch_slot3<0, kPlain ? 1 : 0, MODE>(t);
    if (!kExcl && v.max_sources <= 2) return launch_slot3<0, kExcl ? 0 : 2, MODE>(t);
    if (kPlain && v.max_sources <= 3) return launch_slot3<0, kPlain ? 3 : 0, MODE>(t);
    if (eight) return launch_slot3<0, 8, MODE>(t);
    return launch_slot3<0, 0, MODE>(t);
  }
  if (v.cls_kind == 2) {
    if (v.max_sources <= 2) return launch_slot3<2, 2, MODE>(t);
    if (eight) return launch_slot3<2, 8, MODE>(t);
    return launch_slot3<2, 0, MODE>(t);
  }
  return launch_slot3<1, 0, MODE>(t);
}

int launch_slot_plain(const SlotCall& t);
int launch_slot_excl(const SlotCall& t);
int launch_slot_excl16(const SlotCall& t);
int launch_slot_het(const SlotCall& t);

}  // namespace pe
