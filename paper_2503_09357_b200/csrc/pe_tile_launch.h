// Internal: launch templates of pe_eval_tile_kernel.  The instantiations are spread over one translation unit
// per assignment layout and kernel mode (pe_tile_*.cu) so that they compile in parallel.
#pragma once
#include "pe_kernel_tile.cuh"
#include "pe_launch.h"

namespace pe {

struct TileCall {
  const pe_graph* g;
  const Plan* p;
  int64_t K;
  const uint8_t* assign;
  const uint16_t* order;
  uint32_t flags;
  pe_outputs out;
  cudaStream_t stream;
};

template <int CLS, int EDGES, bool BY_POS, int MODE, int WARPS>
int launch_tile4(const TileCall& t) {
  const Plan& p = *t.p;
  TileShape sh = p.tile;
  sh.vector_init = !BY_POS && sh.lanes % 4 == 0 && t.K % 4 == 0 && ((uintptr_t)t.assign & 3u) == 0;
  auto go = [&](auto kern) -> int {
    if (!set_smem(kern, p.smem)) return PE_ERR_CUDA;
    kern<<<(unsigned)p.grid, p.threads, p.smem, t.stream>>>(t.g->tview, t.g->d_tblob, t.K, t.assign, t.order, t.out,
                                                             t.g->d_error, sh);
    return PE_OK;
  };
  if (!t.out.start) return go(pe_eval_tile_kernel<CLS, EDGES, BY_POS, 0, MODE, WARPS>);
  if (t.flags & PE_TIMES_BY_OP) return go(pe_eval_tile_kernel<CLS, EDGES, BY_POS, 2, MODE, WARPS>);
  return go(pe_eval_tile_kernel<CLS, EDGES, BY_POS, 1, MODE, WARPS>);
}

template <int CLS, int EDGES, bool BY_POS, int MODE>
int launch_tile3(const TileCall& t) {
  // More registers gain nothing for a step with channels (within 3 %), and by position for one with branches or with
  // durations by machine (V = 480 K = 32768 172 us with 128 registers, 178 with more; MoE graph 102 and 109).
  constexpr bool kBoth = MODE != kTileExcl && MODE != kTileExclLong && !(BY_POS && (MODE == kTileHet || CLS == 1 || EDGES == 0));
  if (kBoth && t.p->threads <= 32 * kTileWarps) return launch_tile4<CLS, EDGES, BY_POS, MODE, kBoth ? kTileWarps : 2 * kTileWarps>(t);
  return launch_tile4<CLS, EDGES, BY_POS, MODE, 2 * kTileWarps>(t);
}

// EDGES specialisations (two or three inline edges and nothing else) exist for the modes that carry the main path.
template <bool BY_POS, int MODE>
int launch_tile_mode(const TileCall& t) {
  const PeTileView& v = t.g->tview;
  constexpr bool kSpecial = MODE == kTilePlain || MODE == kTileS16;
  if (v.cls_kind == 0) {
    if (kSpecial && v.max_indeg <= 2) return launch_tile3<0, kSpecial ? 2 : 0, BY_POS, MODE>(t);
    if (kSpecial && v.max_indeg == 3) return launch_tile3<0, kSpecial ? 3 : 0, BY_POS, MODE>(t);
    return launch_tile3<0, 0, BY_POS, MODE>(t);
  }
  if (v.cls_kind == 2) {
    if (kSpecial && v.max_indeg <= 2) return launch_tile3<2, kSpecial ? 2 : 0, BY_POS, MODE>(t);
    return launch_tile3<2, 0, BY_POS, MODE>(t);
  }
  return launch_tile3<1, 0, BY_POS, MODE>(t);
}

int launch_tile_op_plain(const TileCall& t);
int launch_tile_op_s16(const TileCall& t);
int launch_tile_op_excl(const TileCall& t);
int launch_tile_op_het(const TileCall& t);
int launch_tile_op_long(const TileCall& t);
int launch_tile_pos_plain(const TileCall& t);
int launch_tile_pos_s16(const TileCall& t);
int launch_tile_pos_excl(const TileCall& t);
int launch_tile_pos_het(const TileCall& t);
int launch_tile_pos_long(const TileCall& t);

}  // namespace pe
