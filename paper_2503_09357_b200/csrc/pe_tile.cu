// Plan and launcher of pe_eval_tile_kernel (instantiated in pe_tile_*_*.cu).
#include "pe_tile_launch.h"

namespace pe {

namespace {
inline size_t up16(size_t x) { return (x + 15) & ~(size_t)15; }
}

// Block shape: W warps of P lanes that together use the shared memory of an SM.
bool plan_tile(const pe_graph* g, int64_t K, bool by_pos, bool exclusive, Plan* p) {
  if (!g->tile_ok || K >= ((int64_t)1 << 30)) return false;   // (row pitches in bytes are 32-bit)
  if (g->hetero && exclusive) return false;
  const PeTileView& tv = g->tview;
  int jb = 1;
  while ((1 << jb) < g->D) ++jb;
  int mode = kTilePlain;
  if (g->hetero) mode = kTileHet;
  else if (exclusive) mode = kTileExcl;
  else if (jb < 16 && g->time_bound < ((int64_t)1 << (16 - jb)) - 1) mode = kTileS16;
  if (mode != kTileS16 && g->time_bound >= kTileTimeLimit) {
    if (g->hetero || g->time_bound >= kPackedTimeLimit) return false;
    mode = exclusive ? kTileExclLong : kTileLong;
  }
  const size_t fixed = up16((size_t)tv.bytes + 8);
  if (fixed >= g->smem_optin) return false;
  const size_t D = (size_t)g->D, rows = (size_t)g->V + 1;
  auto bytes = [&](size_t W, size_t P) {
    const size_t per = up16(P * 16 * D) + (g->has_weight ? up16(P * 4 * D) : 0) + (exclusive ? up16(P * 4 * D * D) : 0);
    const size_t states = mode == kTileS16 ? (W + 1) / 2 : W;
    return fixed + W * per + states * up16(P * 4 * rows);
  };
  // The time of a round (all resident tiles, V positions) is that of one step as long as every warp has a scheduler to
  // itself and rises from the fifth warp on, more where narrow rows meet in the same banks, and once more beyond
  // kTileWarps, where a step has half the registers; the largest number of candidates per unit of that is taken.
  // Measured, ns a step by W x P (by operator): V = 961 / D = 8 2x24 87, 3x16 84, 4x12 90, 6x8 110, 8x4 111, 12x4 164,
  // 13x4 195; V = 256 / D = 8 3x32 102, 4x32 105, 5x32 129, 6x32 145, 7x28 198, 8x24 186; V = 480, 16-bit words 4x32 105,
  // 5x32 123, 6x32 128, 7x24 140, 8x24 157; V = 64 16x32 51 us in all (K = 200000), 8x32 59.  By-operator machine ids are
  // read four candidates at a time: a width that is no multiple of four costs 40 to 50 % there (V = 961 2x24 87, 2x26 131)
  // and nothing by position (101 and 100; V = 684 / D = 6 3x24 105, 4x19 107).
  const size_t grain = by_pos ? 1 : 4;
  size_t bestW = 0, bestP = 0;
  double best = 0;
  for (size_t W = 1; W <= 2 * kTileWarps; ++W)
    for (size_t P = 32; P >= 4; P -= grain)
      if (bytes(W, P) <= g->smem_optin) {
        double round = W <= 4 ? 1.0 : 1.0 + 0.14 * (double)(W - 4);
        if (W > 4 && P < 32) round /= 0.9;
        if (W > kTileWarps) round /= 0.88;
        const double score = (double)(W * P) / round;
        if (score > best) { best = score; bestW = W; bestP = P; }
        break;
      }
  if (bestW == 0) return false;
  p->tile_resident = (int)(bestW * bestP);
  // no more warps than the batch gives work to, equal rounds for all
  const int64_t tiles = (K + (int64_t)bestP - 1) / (int64_t)bestP;
  const int64_t sms = g->sm_count;
  const int64_t rounds = (tiles + sms * (int64_t)bestW - 1) / (sms * (int64_t)bestW);
  p->tile_rounds = rounds;
  if (rounds > 0) {
    const int64_t w = (tiles + sms * rounds - 1) / (sms * rounds);
    if (w < (int64_t)bestW) bestW = (size_t)w;
  }
  p->variant = PE_VARIANT_SHARED;
  p->compact = true;
  p->tiled = true;
  p->exclusive = exclusive;
  p->tile_mode = mode;
  p->threads = (int)(32 * bestW);
  p->grid = tiles < sms ? tiles : sms;
  p->smem = bytes(bestW, bestP);
  p->workspace = 0;
  TileShape& sh = p->tile;
  sh.lanes = (int)bestP;
  sh.jbits = mode == kTileS16 ? jb : 8;
  sh.tiles = tiles;
  sh.dev_bytes = (uint32_t)up16(bestP * 16 * D);
  sh.wsum_bytes = g->has_weight ? (uint32_t)up16(bestP * 4 * D) : 0;
  sh.chan_bytes = exclusive ? (uint32_t)up16(bestP * 4 * D * D) : 0;
  sh.state_bytes = (uint32_t)up16(bestP * 4 * rows);
  sh.off_dev = (uint32_t)fixed;
  sh.off_wsum = sh.off_dev + (uint32_t)bestW * sh.dev_bytes;
  sh.off_chan = sh.off_wsum + (uint32_t)bestW * sh.wsum_bytes;
  sh.off_state = sh.off_chan + (uint32_t)bestW * sh.chan_bytes;
  return true;
}

int launch_tile(const pe_graph* g, const Plan& p, bool by_pos, int64_t K, const uint8_t* assign, const uint16_t* order,
                uint32_t flags, const pe_outputs& out, cudaStream_t stream) {
  TileCall t;
  t.g = g; t.p = &p; t.K = K; t.assign = assign; t.order = order; t.flags = flags; t.out = out; t.stream = stream;
  switch (p.tile_mode) {
    case kTilePlain: return by_pos ? launch_tile_pos_plain(t) : launch_tile_op_plain(t);
    case kTileS16: return by_pos ? launch_tile_pos_s16(t) : launch_tile_op_s16(t);
    case kTileExcl: return by_pos ? launch_tile_pos_excl(t) : launch_tile_op_excl(t);
    case kTileHet: return by_pos ? launch_tile_pos_het(t) : launch_tile_op_het(t);
    case kTileLong:
    case kTileExclLong: return by_pos ? launch_tile_pos_long(t) : launch_tile_op_long(t);
    default: return PE_ERR_UNSUPPORTED;
  }
}

}  // namespace pe
