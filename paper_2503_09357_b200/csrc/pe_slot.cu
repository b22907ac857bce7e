// Plan and launcher of the slot kernels (pe_eval_slot_kernel is instantiated in pe_slot_*.cu).
#include "pe_slot_launch.h"

#include <algorithm>

namespace pe {

namespace {

inline size_t up16(size_t x) { return (x + 15) & ~(size_t)15; }
inline size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

constexpr size_t kSlotChunkBytes = (size_t)1 << 30;   // workspace of a chunk

size_t gather_smem(const pe_graph* g, bool by_pos, size_t C) {
  const size_t V = (size_t)g->V, D = (size_t)g->D;
  return (by_pos ? 0 : (V + 1) * C) + D * C * 4 * (g->has_weight ? 2 : 1) + (C + 1) * 4;
}

// Candidates a block of the gather and times kernels: wide rows, as long as two blocks fit on an SM.
template <typename Bytes>
size_t tile_width(const pe_graph* g, Bytes bytes) {
  for (const size_t C : {32, 16, 8})
    if (2 * (bytes(C) + 1024) <= g->smem_per_sm) return C;
  for (const size_t C : {16, 8})
    if (bytes(C) <= g->smem_optin) return C;
  return 0;
}

template <int C>
int gather(const pe_graph* g, bool by_pos, int64_t K, int64_t n, const uint8_t* assign, const uint16_t* order, int32_t* busy,
           uint4* entries, int64_t pitch, uint32_t* status, int32_t* wsum, cudaStream_t stream) {
  auto go = [&](auto kern) -> int {
    const size_t smem = gather_smem(g, by_pos, C);
    if (!set_smem(kern, smem)) return PE_ERR_CUDA;
    kern<<<(unsigned)((n + C - 1) / C), kGatherThreads, smem, stream>>>(g->sview, g->d_sblob, K, n, assign, order, busy, entries, pitch, status, wsum);
    return PE_OK;
  };
  const bool vec = K % 4 == 0 && n % 4 == 0 && ((uintptr_t)order & 3u) == 0 && ((uintptr_t)assign & 3u) == 0;
  if (vec) {
    if (g->hetero) return by_pos ? go(pe_slot_gather_kernel<C, true, true, true>) : go(pe_slot_gather_kernel<C, false, true, true>);
    return by_pos ? go(pe_slot_gather_kernel<C, true, false, true>) : go(pe_slot_gather_kernel<C, false, false, true>);
  }
  if (g->hetero) return by_pos ? go(pe_slot_gather_kernel<C, true, true, false>) : go(pe_slot_gather_kernel<C, false, true, false>);
  return by_pos ? go(pe_slot_gather_kernel<C, true, false, false>) : go(pe_slot_gather_kernel<C, false, false, false>);
}

template <int C>
int times_by_op(const pe_graph* g, int64_t K, int64_t n, const uint4* entries, const uint32_t* words, int64_t pitch, int32_t* start,
                int32_t* finish, cudaStream_t stream) {
  auto go = [&](auto kern) -> int {
    const size_t smem = (size_t)(g->V + 1) * C * 4;
    if (!set_smem(kern, smem)) return PE_ERR_CUDA;
    kern<<<(unsigned)((n + C - 1) / C), kGatherThreads, smem, stream>>>(g->sview, g->d_sblob, K, n, entries, words, pitch, start, finish);
    return PE_OK;
  };
  return g->hetero ? go(pe_slot_times_kernel<C, true>) : go(pe_slot_times_kernel<C, false>);
}

}  // namespace

bool plan_slot(const pe_graph* g, int64_t K, uint32_t flags, bool times, Plan* p) {
  if (!g->slot_ok || K >= ((int64_t)1 << 30)) return false;   // (row pitches in bytes are 32-bit)
  const bool by_pos = (flags & PE_ASSIGN_BY_POS) != 0, exclusive = (flags & PE_COMM_EXCLUSIVE) != 0;
  const bool by_op_times = times && (flags & PE_TIMES_BY_OP) != 0;
  if (g->hetero && exclusive) return false;
  const PeSlotView& sv = g->sview;
  // Marks: no kernel with channels.  By operator on one kind of machine such graphs of any size ran without a workspace before
  // there were slot kernels, and programs with large graphs count on that (4 bytes a position and candidate: 268 MB for V = 1024
  // K = 65536); up to 512 operators the workspace is small enough to ask for.  It is no limit of the kernels.  Measured (us, a
  // lane per candidate / slot kernels): taken, V = 484 D = 64 K = 16384 107 / 73, K = 131072 604 / 503; refused, V = 529 D = 64
  // K = 16384 104 / 93, K = 131072 688 / 644, V = 1024 D = 8 K = 65536 807 / 751, V = 1024 D = 64 K = 131072 1960 / 1506,
  // bidirectional pipeline V = 960 K = 131072 1403 / 922.
  if (sv.marks && (exclusive || (!by_pos && !g->hetero && g->V > 512))) return false;
  p->slot_gather = (int)tile_width(g, [&](size_t C) { return gather_smem(g, by_pos, C); });
  p->slot_times = (int)tile_width(g, [&](size_t C) { return (size_t)(g->V + 1) * C * 4; });
  if (p->slot_gather == 0 || p->slot_times == 0) return false;
  const int mode = g->hetero ? kSlotHet : (!exclusive ? kSlotPlain : (g->time_bound < 65536 ? kSlotExcl16 : kSlotExcl));
  const size_t fixed = up16((size_t)sv.bytes + 8), D = (size_t)g->D, rows = (size_t)sv.nslots + 2;
  const size_t chan = exclusive ? (D * D + 1) * (mode == kSlotExcl16 ? 2 : 4) : 0;
  auto bytes = [&](size_t W, size_t P) { return fixed + W * (P * 16 * kSlotQuads + up16(P * 8 * D) + up16(P * chan) + up16(P * 4 * rows)); };
  size_t bestW = 0, bestP = 0;
  double best = 0;
  for (size_t W = 1; W <= (size_t)kSlotWarps; ++W)
    for (size_t P = 32; P >= 4; P -= 4)
      if (bytes(W, P) <= g->smem_optin) {
        // (from seven warps on a step takes the longer the more there are)
        const double score = (double)(W * P) / std::max(1.0, (double)W / 7.0) * (1.0 + 1e-3 * (double)W);
        if (score > best) { best = score; bestW = W; bestP = P; }
        break;
      }
  if (bestW == 0) return false;
  p->tile_resident = (int)(bestW * bestP);
  const int64_t sms = g->sm_count, wave = sms * (int64_t)(bestW * bestP);
  const size_t per = up16((size_t)g->V * 4) + 4 + (g->has_weight ? D * 4 : 0) + (by_op_times ? (size_t)g->V * 4 : 0);   // workspace of a candidate
  int64_t chunk = (int64_t)(kSlotChunkBytes / per) / wave * wave;
  if (chunk < wave) chunk = wave;
  if (chunk > K) chunk = K;
  const int64_t pitch = (chunk + 31) / 32 * 32;
  p->slot_chunk = chunk;
  p->slot_pitch = pitch;
  size_t at = up256((size_t)pitch * 16 * (((size_t)g->V + 3) / 4));
  p->slot_off_status = at; at = up256(at + (size_t)pitch * 4);
  p->slot_off_wsum = at;   at = up256(at + (g->has_weight ? (size_t)pitch * 4 * D : 0));
  p->slot_off_words = at;  at = up256(at + (by_op_times ? (size_t)pitch * 4 * (size_t)g->V : 0));
  p->workspace = at;
  // no more warps than a chunk gives work to, equal rounds for all
  const int64_t tiles = (chunk + (int64_t)bestP - 1) / (int64_t)bestP;
  const int64_t rounds = (tiles + sms * (int64_t)bestW - 1) / (sms * (int64_t)bestW);
  if (rounds > 0) {
    const int64_t w = (tiles + sms * rounds - 1) / (sms * rounds);
    if (w < (int64_t)bestW) bestW = (size_t)w;
  }
  p->tile_rounds = chunk > 0 ? rounds * (K / chunk) + (K % chunk + wave - 1) / wave : 0;
  p->variant = PE_VARIANT_SHARED;
  p->compact = true;
  p->slot = true;
  p->exclusive = exclusive;
  p->tile_mode = mode;
  p->threads = (int)(32 * bestW);
  p->smem = bytes(bestW, bestP);
  SlotShape& sh = p->slot_shape;
  sh.lanes = (int)bestP;
  sh.tiles = 0;
  sh.dev_bytes = (uint32_t)up16(bestP * 8 * D);
  sh.chan_bytes = (uint32_t)up16(bestP * chan);
  sh.state_bytes = (uint32_t)up16(bestP * 4 * rows);
  sh.off_ring = (uint32_t)fixed;
  sh.off_dev = sh.off_ring + (uint32_t)(bestW * bestP * 16 * kSlotQuads);
  sh.off_chan = sh.off_dev + (uint32_t)bestW * sh.dev_bytes;
  sh.off_state = sh.off_chan + (uint32_t)bestW * sh.chan_bytes;
  return true;
}

int launch_slot(const pe_graph* g, const Plan& p, bool by_pos, int64_t K, const uint8_t* assign, const uint16_t* order,
                uint32_t flags, const pe_outputs& out, void* workspace, cudaStream_t stream, int64_t* launches) {
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  uint4* entries = reinterpret_cast<uint4*>(ws);
  uint32_t* status = reinterpret_cast<uint32_t*>(ws + p.slot_off_status);
  int32_t* wsum = g->has_weight ? reinterpret_cast<int32_t*>(ws + p.slot_off_wsum) : nullptr;
  uint32_t* words = out.start && (flags & PE_TIMES_BY_OP) ? reinterpret_cast<uint32_t*>(ws + p.slot_off_words) : nullptr;
  for (int64_t c0 = 0; c0 < K; c0 += p.slot_chunk) {
    const int64_t n = std::min(p.slot_chunk, K - c0);
    int32_t* busy = out.busy ? out.busy + c0 : nullptr;
    const int64_t pitch = p.slot_pitch;
    int rc = PE_ERR_UNSUPPORTED;
    switch (p.slot_gather) {
      case 32: rc = gather<32>(g, by_pos, K, n, assign + c0, order + c0, busy, entries, pitch, status, wsum, stream); break;
      case 16: rc = gather<16>(g, by_pos, K, n, assign + c0, order + c0, busy, entries, pitch, status, wsum, stream); break;
      case 8: rc = gather<8>(g, by_pos, K, n, assign + c0, order + c0, busy, entries, pitch, status, wsum, stream); break;
    }
    if (rc != PE_OK) return rc;
    SlotCall t;
    t.g = g; t.p = &p; t.K = K; t.n = n; t.pitch = pitch;
    t.entries = entries; t.status = status; t.wsum = wsum; t.words = words;
    t.shape = p.slot_shape;
    t.shape.tiles = (n + t.shape.lanes - 1) / t.shape.lanes;
    t.grid = std::min<int64_t>(t.shape.tiles, g->sm_count);
    t.out = out;
    if (out.start) { t.out.start = out.start + c0; t.out.finish = out.finish + c0; }
    if (out.makespan) t.out.makespan = out.makespan + c0;
    if (out.peak_mem) t.out.peak_mem = out.peak_mem + c0;
    if (out.status) t.out.status = out.status + c0;
    t.stream = stream;
    switch (p.tile_mode) {
      case kSlotPlain: rc = launch_slot_plain(t); break;
      case kSlotExcl: rc = launch_slot_excl(t); break;
      case kSlotExcl16: rc = launch_slot_excl16(t); break;
      case kSlotHet: rc = launch_slot_het(t); break;
      default: rc = PE_ERR_UNSUPPORTED;
    }
    if (rc != PE_OK) return rc;
    *launches += 2;
    if (words) {
      int32_t *start = out.start + c0, *finish = out.finish + c0;
      switch (p.slot_times) {
        case 32: rc = times_by_op<32>(g, K, n, entries, words, pitch, start, finish, stream); break;
        case 16: rc = times_by_op<16>(g, K, n, entries, words, pitch, start, finish, stream); break;
        case 8: rc = times_by_op<8>(g, K, n, entries, words, pitch, start, finish, stream); break;
        default: rc = PE_ERR_UNSUPPORTED;
      }
      if (rc != PE_OK) return rc;
      *launches += 1;
    }
  }
  return PE_OK;
}

}  // namespace pe
