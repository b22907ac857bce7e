// Variant SHARED over the tile encoding: one lane per candidate, everything on chip.
//
// A warp evaluates a tile of P <= 32 candidates, lane l the candidate c0 + l, and then takes the next
// tile; the warps of a block are independent of each other (no block barrier after the graph has been
// staged), so the initial pass of one tile overlaps the main loop of the others and a small batch
// spreads over the SMs a warp at a time.
//
// What bounds it: the recurrence.  Position k + 1 may need the end time that position k has just
// written, so a step costs one shared-memory round trip (state words and machine record, ~30 cycles)
// plus the maximum over the sources, the duration and the store; shared memory holds few candidates
// (4 V bytes each), so few warps hide that latency, and every instruction of a step counts.  Hence:
//   * everything of position k + 1 that does not depend on a time is fetched during step k (operator
//     record, own machine, link-class row, duration by machine), order entries kRing positions ahead
//     into a register ring that is refilled in place;
//   * times are kept and compared in packed form, time << jb | machine.  A maximum over packed words is
//     a maximum over times (the machine bits only break ties), so a source costs: address, load,
//     same-machine test, delay select, fused add-max;
//   * validity costs one instruction a step: an operator that is not scheduled yet holds a time field
//     beyond every reachable time, which reaches the machine's last end time; a repeated operator does not
//     find exactly the unscheduled word (behind a missing source it finds a later time, so a comparison with
//     scheduled words alone would let repetitions add up until the packed time wraps); an entry that is no
//     operator is clamped to the sentinel row V, which counts as scheduled.
// Measured on B200 (before: the thread-per-candidate kernel this one replaces, 92 instructions and ~370 cycles a
// step at V = 256; now 68 and ~230): V = 256 / D = 8, K = 2^20: 1.85 -> 1.19 ms; bidirectional pipeline (V = 480),
// K = 65536: 352 -> 166 us, with durations by machine, K = 16384: 490 -> 113 us (generic kernel before); multi-modal
// graph K = 65536: 3.34 -> 2.42 ms (warp per candidate), with exclusive channels, K = 16384: 2.74 -> 1.75 ms
// (global-state kernel before).
//
// State word: uint32_t time << 8 | machine, or uint16_t time << jb | machine when the graph's time bound
// and machine count fit 16 bits (two warps then share the 32-bit words of a row, one the low and one the
// high halves, so the lanes of a warp still fall into different banks).  Tile layout [operator][P].
// Per-machine record {free (packed), busy, level, peak}, 16 bytes, [machine][P].
#pragma once
#include <type_traits>

#include "pe_device.cuh"
#include "pe_smem.cuh"
#include "pe_tile_shape.h"

namespace pe {

constexpr int64_t kTileTimeLimit = 0x7FFFFF;        // 32-bit words: end times stay below this
constexpr uint32_t kTileUnscheduled = 0x7FFFFF00u;  // | machine; sums with a delay and a duration do not wrap
// Longer times leave no room above them: such a sum may wrap, so the words of the sources themselves are tested.
constexpr uint32_t kTileUnscheduledLong = 0xFFFFFF00u;

// Order entries and by-position machine ids: volatile, so that a block's requests stay in front of its steps.
__device__ __forceinline__ uint32_t ldg_u16(const void* p) {
  uint16_t v;
  asm volatile("ld.global.nc.u16 %0, [%1];" : "=h"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ uint32_t ldg_u8(const void* p) {
  uint32_t v;
  asm volatile("ld.global.nc.u8 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}

// CLS: 0 = one link class, every pair connected; 1 = class table in shared memory (one or two classes,
// pairs without a channel possible); 2 = two classes, every pair connected, at most 32 machines: the class
// of a pair is a bit of a row word.
// EDGES: 2 / 3 = no operator has more incoming edges, all inline; 0 = inline edges, then the edge list.
// TIMES: 0 = none, 1 = by position, 2 = by operator.
// WARPS: largest number of warps of a block.  With kTileWarps a thread may use the registers that a request block of
// sixteen positions needs without spilling (128 registers and 4 to 12 bytes of spills with twice as many warps: V = 1024 /
// D = 64 K = 65536 1110 -> 1038 us by operator and, with blocks of 16 instead of 8, 1178 -> 954 by position; multi-modal
// graph 2434 -> 2310 and 2337 -> 2121; V = 256 / D = 8 K = 2^20 1205 -> 1163 and 1249 -> 1032).
template <int CLS, int EDGES, bool BY_POS, int TIMES, int MODE, int WARPS>
__global__ void __launch_bounds__(32 * WARPS) pe_eval_tile_kernel(PeTileView g, const uint8_t* __restrict__ blob, int64_t K,
                                                           const uint8_t* __restrict__ assign,
                                                           const uint16_t* __restrict__ order, pe_outputs out, int* err,
                                                           TileShape sh) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  constexpr uint32_t FULL = 0xFFFFFFFFu;
  constexpr bool S16 = MODE == kTileS16, EXCL = MODE == kTileExcl || MODE == kTileExclLong, HET = MODE == kTileHet;
  constexpr bool LONG = MODE == kTileLong || MODE == kTileExclLong;
  constexpr uint32_t kUnsched32 = LONG ? kTileUnscheduledLong : kTileUnscheduled;
  using StateT = typename std::conditional<S16, uint16_t, uint32_t>::type;
  // Order entries (and by-position machine ids) per request.  A step with branches, or with channels or durations by
  // machine, is so long that sixteen of them are no longer inlined or overflow the instruction cache.
  constexpr bool kRoomy = WARPS <= kTileWarps, kStraight = !EXCL && !HET && CLS != 1 && EDGES != 0;
  constexpr bool kEight = kRoomy ? !kStraight || (BY_POS && TIMES == 1 && CLS == 0 && EDGES == 2 && !S16) : BY_POS || EXCL || HET;
  constexpr int kRing = kEight ? 8 : 16;
  // Whether a step carries stores that are never executed (see there).
  constexpr bool kIdleStores = kRoomy && kStraight && TIMES != 1 && !(TIMES == 0 && !BY_POS && CLS == 0 && (S16 || EDGES == 2));
  constexpr int NIN = CLS == 0 ? (EDGES == 2 ? 2 : 3) : 2;   // edges that the record carries inline
  const int V = g.V, D = g.D;
  const int lane = threadIdx.x & 31;
  const int warp = __shfl_sync(FULL, (int)(threadIdx.x >> 5), 0);
  const int nwarps = blockDim.x >> 5;
  const int P = sh.lanes;
  const uint32_t jb = S16 ? (uint32_t)sh.jbits : 8u;
  const uint32_t jmask = (1u << jb) - 1u;
  const uint32_t unsched = S16 ? ((0xFFFFu >> jb) << jb) : kUnsched32;

  {
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw + g.bytes);
    if (!stage_blob(smem_raw, blob, g.bytes, bar, err)) return;
  }
  if (S16) {   // delays and durations in units of the packed time field, once per block
    uint4* recs_w = reinterpret_cast<uint4*>(smem_raw + g.ops);
    for (int i = threadIdx.x; i <= V; i += blockDim.x) {
      uint4 r = recs_w[i];
      auto hi = [&](uint32_t x) { return ((x >> 16) << (jb + 16)) | (x & 0xFFFFu); };
      auto both = [&](uint32_t x) { return ((x >> 16) << (jb + 16)) | ((x << jb) & 0xFFFFu); };
      const int n = (int)((r.x >> 16) & 0xFFu);
      r.x = (r.x & 0xFFFF0000u) | ((r.x << jb) & 0xFFFFu);
      if (CLS == 0) {
        r.y = hi(r.y); r.z = hi(r.z);
        if (n <= 3) r.w = hi(r.w);
      } else {
        r.z = both(r.z); r.w = both(r.w);
      }
      recs_w[i] = r;
    }
    if (EDGES == 0) {
      if (CLS == 0) {
        uint32_t* ed = reinterpret_cast<uint32_t*>(smem_raw + g.edges);
        for (int q = threadIdx.x; q < g.list_edges; q += blockDim.x) ed[q] = ((ed[q] >> 16) << (jb + 16)) | (ed[q] & 0xFFFFu);
      } else {
        uint2* ed = reinterpret_cast<uint2*>(smem_raw + g.edges);
        for (int q = threadIdx.x; q < g.list_edges; q += blockDim.x)
          ed[q].y = ((ed[q].y >> 16) << (jb + 16)) | ((ed[q].y << jb) & 0xFFFFu);
      }
    }
    __syncthreads();
  }
  const int32_t* weight = g.has_weight ? reinterpret_cast<const int32_t*>(smem_raw + g.weight) : nullptr;
  const int32_t* cap = reinterpret_cast<const int32_t*>(smem_raw + g.cap);

  const uint32_t pitch = (uint32_t)P * 4u;   // bytes of a row of words
  const int ml = lane < P ? lane : P - 1;    // (lanes beyond the tile have no column: they only copy, and sit out the main loop)
  const uint32_t vlast = (uint32_t)V, dmax = (uint32_t)(D - 1);
  uint8_t* st_base = S16 ? smem_raw + sh.off_state + (uint32_t)(warp >> 1) * sh.state_bytes + (uint32_t)ml * 4u + (uint32_t)(warp & 1) * 2u
                         : smem_raw + sh.off_state + (uint32_t)warp * sh.state_bytes + (uint32_t)ml * 4u;
  uint8_t* dv_base = smem_raw + sh.off_dev + (uint32_t)warp * sh.dev_bytes + (uint32_t)ml * 16u;
  uint8_t* ws_base = smem_raw + sh.off_wsum + (uint32_t)warp * sh.wsum_bytes + (uint32_t)ml * 4u;
  uint8_t* ch_base = smem_raw + sh.off_chan + (uint32_t)warp * sh.chan_bytes + (uint32_t)ml * 4u;
  auto state = [&](uint32_t p) -> StateT& { return *reinterpret_cast<StateT*>(st_base + p * pitch); };
  auto dev = [&](uint32_t j) -> int4& { return *reinterpret_cast<int4*>(dv_base + j * (pitch * 4u)); };
  const uint32_t smem_a = smem_u32(smem_raw);
  const uint32_t rec_a = smem_a + g.ops, cls_a = smem_a + g.cls, row_a = smem_a + g.cls_row, durm_a = smem_a + g.durm;
  const uint32_t st_a = smem_u32(st_base), dv_a = smem_u32(dv_base), ch_a = smem_u32(ch_base);
  const uint32_t dpitch = pitch * 4u;

  const uint32_t K2 = (uint32_t)K * 2u, K4 = (uint32_t)K * 4u, K1 = (uint32_t)K;   // row pitches in bytes (K < 2^26)

  for (int64_t tile = (int64_t)warp * gridDim.x + blockIdx.x; tile < sh.tiles; tile += (int64_t)nwarps * gridDim.x) {
    const int64_t c0 = tile * P;
    const int in_tile = (int)(K - c0 < P ? K - c0 : P);
    const bool cand = lane < in_tile;
    const uint32_t cc = (uint32_t)c0 + (uint32_t)(lane < in_tile ? lane : in_tile - 1);   // (a lane without a candidate re-does the last one)
    const bool write = lane < P;

    const uint8_t* ord_b = reinterpret_cast<const uint8_t*>(order) + (size_t)cc * 2;   // row of the next block to prefetch
    const uint8_t* asg_b = assign + cc;
    uint32_t ring[kRing], aring[kRing];
#pragma unroll
    for (int u = 0; u < kRing; ++u) {
      const uint32_t row = (uint32_t)min(u, V - 1);
      ring[u] = *reinterpret_cast<const uint16_t*>(ord_b + (size_t)row * K2);
      if (BY_POS) aring[u] = asg_b[(size_t)row * K1];
    }

    // ---- initial pass: unscheduled, machine of every operator (by-operator assignments) ----
    __syncwarp();
    uint32_t raw_bad = 0;
    if (BY_POS) {
      if (write)
        for (int i = 0; i < V; ++i) state((uint32_t)i) = (StateT)unsched;
    } else if (sh.vector_init && in_tile == P) {
      // four candidates of a row per load; consecutive groups of P / 4 lanes take consecutive rows
      const int wpr = P >> 2, rpi = 32 / wpr;
      const int r = lane / wpr, cw = lane - r * wpr;
      const bool mine = r < rpi;
      const uint32_t d4 = dmax * 0x01010101u;
      const uint8_t* src = assign + c0 + 4 * cw;
      const uint32_t words_a = st_a - (uint32_t)ml * 4u + (uint32_t)cw * 16u;
      if constexpr (!S16) {
        // All rows are in flight at once: the raw bytes land in the last quarter of the tile's own state area and
        // are expanded in place from the front; the words of a row never reach the bytes of a later row.
        const uint32_t bytes_a = st_a - (uint32_t)ml * 4u + (uint32_t)(V + 1) * pitch - (uint32_t)(V * P) + (uint32_t)cw * 4u;
        if (mine)
          for (int row = r; row < V; row += rpi) cp_async4(bytes_a + (uint32_t)(row * P), src + (size_t)row * (size_t)K);
        cp_async_wait_all();
        __syncwarp();
        constexpr int kBatch = 4;
        for (int r0 = r; r0 < V + r; r0 += kBatch * rpi) {
          uint32_t x[kBatch];
#pragma unroll
          for (int q = 0; q < kBatch; ++q) {
            const int row = r0 + q * rpi;
            x[q] = lds32(bytes_a + (uint32_t)(min(row, V - 1) * P));
          }
          __syncwarp();
#pragma unroll
          for (int q = 0; q < kBatch; ++q) {
            const int row = r0 + q * rpi;
            const uint32_t xc = __vminu4(x[q], d4);
            raw_bad |= x[q] ^ xc;
            if (mine && row < V)
              sts128(words_a + (uint32_t)row * pitch,
                     make_uint4(__byte_perm(xc, kUnsched32, 0x7650), __byte_perm(xc, kUnsched32, 0x7651),
                                __byte_perm(xc, kUnsched32, 0x7652), __byte_perm(xc, kUnsched32, 0x7653)));
          }
          __syncwarp();
        }
      } else {   // (the words belong to two warps: nothing else may land between them)
        constexpr int kBatch = 16;
        for (int r0 = r; r0 < V + r; r0 += kBatch * rpi) {
          uint32_t x[kBatch];
#pragma unroll
          for (int q = 0; q < kBatch; ++q) {
            const int row = r0 + q * rpi;
            x[q] = *reinterpret_cast<const uint32_t*>(src + (size_t)(mine ? min(row, V - 1) : 0) * (size_t)K);
          }
#pragma unroll
          for (int q = 0; q < kBatch; ++q) {
            const int row = r0 + q * rpi;
            const uint32_t xc = __vminu4(x[q], d4);
            raw_bad |= x[q] ^ xc;
            if (mine && row < V) {
              const uint32_t at = words_a + (uint32_t)row * pitch;
              sts_state<true>(at, unsched | (xc & 0xFFu));
              sts_state<true>(at + 4u, unsched | ((xc >> 8) & 0xFFu));
              sts_state<true>(at + 8u, unsched | ((xc >> 16) & 0xFFu));
              sts_state<true>(at + 12u, unsched | (xc >> 24));
            }
          }
        }
      }
    } else {
      constexpr int kBatch = 16;
      const uint8_t* src = assign + cc;
      for (int i = 0; i < V; i += kBatch) {
        uint32_t x[kBatch];
#pragma unroll
        for (int q = 0; q < kBatch; ++q) x[q] = i + q < V ? (uint32_t)src[(size_t)(i + q) * (size_t)K] : 0u;
#pragma unroll
        for (int q = 0; q < kBatch; ++q) {
          raw_bad |= x[q] > dmax ? 1u : 0u;
          if (i + q < V && write) state((uint32_t)(i + q)) = (StateT)(unsched | min(x[q], dmax));
        }
      }
    }
    if (write) {
      state(vlast) = (StateT)0;
      for (int j = 0; j < D; ++j) dev((uint32_t)j) = make_int4(0, 0, 0, 0);
      if (weight)
        for (int j = 0; j < D; ++j) *reinterpret_cast<int32_t*>(ws_base + (uint32_t)j * pitch) = 0;
      if (EXCL)
        for (int q = 0; q < D * D; ++q) *reinterpret_cast<uint32_t*>(ch_base + (uint32_t)q * pitch) = 0u;
    }
    __syncwarp();

    if (!BY_POS) {   // the next tile's machine ids come from L2 when their turn comes
      const int64_t c_next = c0 + (int64_t)P * nwarps * gridDim.x;
      if (c_next < K)
        for (int row = lane; row < V; row += 32)
          asm volatile("prefetch.global.L2 [%0];" ::"l"(assign + (size_t)row * (size_t)K + (size_t)c_next));
    }

    // ---- main loop ----
    uint32_t st = 0;
    uint32_t src_max = 0;                // LONG: largest word of a source
    uint32_t own_max = 0, dev_max = 0;   // own_max: the word a position finds for its operator, less `unsched`
    uint8_t* start_b = reinterpret_cast<uint8_t*>(out.start) + (size_t)cc * 4;     // this position's row
    uint8_t* finish_b = reinterpret_cast<uint8_t*>(out.finish) + (size_t)cc * 4;

    uint32_t i_cur = min(ring[0], vlast);
    uint4 rec = lds128(rec_a + i_cur * 16u);
    uint32_t own = lds_state<S16>(st_a + i_cur * pitch);
    uint32_t a_cur = BY_POS ? aring[0] : 0u;

    // One position.  o_next / a_next: order entry and by-position machine of the next one.
    auto step = [&](const uint32_t o_next, const uint32_t a_next) {
      const uint32_t i = i_cur;
      uint32_t j;
      if (BY_POS) {
        dev_max = max(dev_max, a_cur);
        j = min(a_cur, dmax);
      } else {
        j = own & jmask;
      }
      const uint4 r4 = rec;
      // sources and machine record: the loads that the previous step's stores may feed
      uint32_t p[NIN], w[NIN];
      if (CLS == 0) {
        p[0] = r4.y & 0xFFFFu;
        p[1] = r4.z & 0xFFFFu;
        if (NIN == 3) p[NIN - 1] = (EDGES == 0 && ((r4.x >> 16) & 0xFFu) > 3u) ? vlast : (r4.w & 0xFFFFu);
      } else {
        p[0] = r4.y & 0xFFFFu;
        p[1] = r4.y >> 16;
      }
#pragma unroll
      for (int q = 0; q < NIN; ++q) w[q] = lds_state<S16>(st_a + p[q] * pitch);
      const uint4 dv = lds128(dv_a + j * dpitch);
      uint32_t crow = 0;
      if (CLS == 2) crow = lds32(row_a + j * 4u);
      uint32_t dur_het = 0;
      if (HET) dur_het = lds16(durm_a + (i * (uint32_t)D + j) * 2u);
      if (BY_POS) own = lds_state<S16>(st_a + i * pitch);
      own_max = max(own_max, own - unsched);
      // the next position's operator
      const uint32_t i_n = min(o_next, vlast);
      const uint4 rec_n = lds128(rec_a + i_n * 16u);
      uint32_t own_n = 0;
      if (!BY_POS) own_n = lds_state<S16>(st_a + i_n * pitch);

      auto pick = [&](uint32_t dd, uint32_t hi) -> uint32_t {   // packed delay: high or low half of dd
        if (S16) return hi ? dd >> 16 : dd & 0xFFFFu;
        return hi ? __byte_perm(dd, 0u, 0x4324) : __byte_perm(dd, 0u, 0x4104);
      };
      // one source: its packed end time plus the delay that applies (Eqs. 11-13)
      auto source = [&](uint32_t pp, uint32_t ww, uint32_t dd) -> uint32_t {
        if (LONG) src_max = max(src_max, ww);
        const bool same = ((ww ^ j) & jmask) == 0u;
        uint32_t d;
        bool channel = true;
        if (CLS == 0) {
          d = pick(dd, 1u);
        } else if (CLS == 2) {
          d = pick(dd, __funnelshift_r(crow, crow, S16 ? ww & jmask : ww) & 1u);   // (shift amount modulo 32)
        } else {
          const uint32_t cl = lds8(cls_a + min(ww & jmask, dmax) * (uint32_t)D + j);
          d = pick(dd, cl == 1u ? 1u : 0u);
          if (cl == 0xFFu) {
            d = 0u;
            channel = false;
            if (!same && pp != vlast) st |= PE_STATUS_NO_CHANNEL;
          }
        }
        if (EXCL) {
          // the transfer starts when its source has ended (Eq. 13) and the channel is free (Eq. 14), lasts D^c (Eq. 11)
          if (!same && pp != vlast && channel) {
            const uint32_t ch = ch_a + (min(ww & 0xFFu, dmax) * (uint32_t)D + j) * pitch;
            const uint32_t t_end = max(ww & ~0xFFu, lds32(ch)) + d;
            sts_state<false>(ch, t_end);
            return t_end;
          }
          return ww;
        }
        return ww + (same ? 0u : d);
      };
      uint32_t r = dv.x;
      if (CLS == 0) {
        const uint32_t t0 = source(p[0], w[0], r4.y), t1 = source(p[1], w[1], r4.z);   // in edge-list order
        r = max(max(t0, t1), r);
        if (NIN == 3) r = max(r, source(p[NIN - 1], w[NIN - 1], r4.w));
        if (EDGES == 0) {
          const uint32_t n = (r4.x >> 16) & 0xFFu;
          if (n > 3u) {
            const uint32_t* ed = reinterpret_cast<const uint32_t*>(smem_raw + g.edges) + r4.w;
            for (uint32_t q = 2; q < n; ++q) r = max(r, source(ed[q] & 0xFFFFu, lds_state<S16>(st_a + (ed[q] & 0xFFFFu) * pitch), ed[q]));
          }
        }
      } else {
        const uint32_t t0 = source(p[0], w[0], r4.z), t1 = source(p[1], w[1], r4.w);
        r = max(max(t0, t1), r);
        if (EDGES == 0) {
          const uint32_t n = (r4.x >> 16) & 0xFFu;
          if (n > 2u) {
            const uint2* ed = reinterpret_cast<const uint2*>(smem_raw + g.edges) + reinterpret_cast<const uint32_t*>(smem_raw + g.slot)[min(i, vlast - 1u)];
            for (uint32_t q = 2; q < n; ++q) r = max(r, source(ed[q].x, lds_state<S16>(st_a + ed[q].x * pitch), ed[q].y));
          }
        }
      }
      // D^o and the machine in packed form (Eq. 3)
      const uint32_t durj = HET ? (dur_het << 8) | j : (S16 ? (r4.x & 0xFFFFu) | j : __byte_perm(r4.x, j, 0x5104));
      const uint32_t rt = r & ~jmask;
      const uint32_t e = rt + durj;
      const int32_t lv = __dp4a((int32_t)r4.x, 0x01000000, (int32_t)dv.z);                      // + A_i (byte 3)
      const uint32_t bz = HET ? dv.y + dur_het : __dp2a_lo(r4.x, 1u, dv.y);                     // + D^o_i (low half)
      sts_state<S16>(st_a + i * pitch, e);
      sts128(dv_a + j * dpitch, make_uint4(e, bz, (uint32_t)lv, (uint32_t)max((int32_t)dv.w, lv)));
      if (kIdleStores)
        // Without any store to global memory in the step the compiler lets the block's requests share a scoreboard with
        // the step's shared-memory loads, and every block waits for DRAM; with a store, executed or not, it does not.
        // Measured (us, without / with): V = 1024 / D = 64 K = 32768 by position 630 / 541, times by operator 950 / 807;
        // multi-modal graph K = 30000 by operator 1360 / 1163, by position 1378 / 1014; bidirectional pipeline K = 65536
        // by position 172 / 133.  (Left out of the forms where it costs: V = 480 by operator 137 / 145.)
        asm volatile("{.reg .pred p; setp.lt.s32 p, %3, 0; @p st.global.u32 [%0], %1; @p st.global.u32 [%0], %2;}"
                     ::"l"(start_b), "r"(rt), "r"(e), "r"(sh.lanes) : "memory");
      if (TIMES == 1) {
        *reinterpret_cast<int32_t*>(start_b) = (int32_t)(rt >> jb);
        *reinterpret_cast<int32_t*>(finish_b) = (int32_t)(e >> jb);
        start_b += K4;
        finish_b += K4;
      }
      if (!BY_POS) {   // a repetition right behind: its own word was read before this step's store
        if (i_n == i) own_n = 0u;
        own = own_n;
      }
      i_cur = i_n;
      rec = rec_n;
      a_cur = a_next;
    };

    // The next block's order entries are requested together at the start of a block: a wait for one load waits
    // for every load that shares its scoreboard (a warp has six), so loads spread over the steps would be waited
    // for a step or two after they were issued.  Measured at V = 256, D = 8 (K = 2^20): entries requested one a
    // step 1583 us, blocks of 16 1242 us, two alternating register sets of 8 1558 us; entries brought to a shared ring by asynchronous
    // copies 1517 us (11 more instructions a step).  With exclusive channels or durations by machine the step is so
    // long that sixteen of them unrolled overflow the instruction cache: blocks of 8 (238 -> 185 us and 138 -> 113 us on
    // the bidirectional pipeline, K = 16384).
    // Lanes beyond the tile stay out: they would read and write the last lane's words, and after a branch nothing keeps
    // them in step with it.
    for (int kb = write ? 0 : V; kb < V; kb += kRing) {
      ord_b += (size_t)kRing * K2;
      asg_b += (size_t)kRing * K1;
      uint32_t nxt[kRing], anxt[kRing];
      if (kb + 2 * kRing <= V) {
#pragma unroll
        for (int u = 0; u < kRing; ++u) {
          nxt[u] = ldg_u16(ord_b + (size_t)u * K2);
          anxt[u] = BY_POS ? ldg_u8(asg_b + (size_t)u * K1) : 0u;
        }
      } else {   // rows that do not exist are not read
#pragma unroll
        for (int u = 0; u < kRing; ++u) {
          const bool have = kb + kRing + u < V;
          nxt[u] = have ? ldg_u16(ord_b + (size_t)u * K2) : 0u;
          anxt[u] = BY_POS && have ? ldg_u8(asg_b + (size_t)u * K1) : 0u;
        }
      }
      if (kb + kRing <= V) {
#pragma unroll
        for (int u = 0; u < kRing; ++u) {
          if (u + 1 < kRing) step(ring[(u + 1) % kRing], BY_POS ? aring[(u + 1) % kRing] : 0u);
          else step(nxt[0], anxt[0]);
        }
      } else {
#pragma unroll
        for (int u = 0; u < kRing - 1; ++u) {
          if (kb + u >= V) break;
          step(ring[u + 1], BY_POS ? aring[u + 1] : 0u);
        }
      }
#pragma unroll
      for (int u = 0; u < kRing; ++u) { ring[u] = nxt[u]; if (BY_POS) aring[u] = anxt[u]; }
    }

    // The lanes that sat out come back.  The loop wrote its words through asm that names no memory; the results read them
    // through ordinary loads.
    __syncwarp();

    // ---- results of the tile ----
    if (TIMES == 2) {
      // Times by operator: the state words hold every end time, so they leave row by row here; a store per step would
      // touch 32 rows at once (bidirectional pipeline K = 65536: 879 -> 212 us; V = 256 / D = 8 K = 2^20: 9.2 -> 1.6 ms).
#pragma unroll 4
      for (int i = 0; i < V; ++i) {
        const uint32_t w = lds_state<S16>(st_a + (uint32_t)i * pitch), d16 = lds32(rec_a + (uint32_t)i * 16u) & 0xFFFFu;
        const int32_t fin = (int32_t)(w >> jb);
        const int32_t d = HET ? (int32_t)lds16(durm_a + ((uint32_t)i * (uint32_t)D + min(w & jmask, dmax)) * 2u) : (int32_t)(S16 ? d16 >> jb : d16);
        if (cand) {
          *reinterpret_cast<int32_t*>(start_b) = fin - d;
          *reinterpret_cast<int32_t*>(finish_b) = fin;
        }
        start_b += K4;
        finish_b += K4;
      }
    }
    if (own_max > jmask) st |= PE_STATUS_ORDER_INVALID;   // an operator twice, or an entry that is no operator
    // a machine's end times rise: the largest last one is the makespan (formed here, not in the loop below: 1185 against
    // 1248 us at V = 256, D = 8)
    uint32_t z = 0;
    for (int j = 0; j < D; ++j) z = max(z, (uint32_t)dev((uint32_t)j).x);
    if ((LONG ? src_max : z) >= unsched) st |= PE_STATUS_ORDER_INVALID;   // an operator ahead of one of its predecessors
    if (BY_POS) {
      if (dev_max > dmax) st |= PE_STATUS_ASSIGN_RANGE;
      // entries at positions that hold no operator are not consulted
      if (dev_max > dmax && own_max > jmask) {
        st &= ~(uint32_t)PE_STATUS_ASSIGN_RANGE;
        for (int k = 0; k < V; ++k)
          if ((uint32_t)order[(size_t)k * (size_t)K + cc] < (uint32_t)V && (uint32_t)assign[(size_t)k * (size_t)K + cc] > dmax)
            st |= PE_STATUS_ASSIGN_RANGE;
      }
    } else if (__any_sync(FULL, raw_bad != 0)) {
      // some machine id of the tile was out of range and clamped: due where the operator is consulted
      for (int k = 0; k < V; ++k) {
        const uint32_t iu = order[(size_t)k * (size_t)K + cc];
        if (iu < (uint32_t)V && (uint32_t)assign[(size_t)iu * (size_t)K + cc] > dmax) st |= PE_STATUS_ASSIGN_RANGE;
      }
    }
    if (weight && write)   // resident weights: the machine of every operator is in its state word
      for (int i = 0; i < V; ++i)
        *reinterpret_cast<int32_t*>(ws_base + min((uint32_t)state((uint32_t)i) & jmask, dmax) * pitch) += weight[i];
    for (int j = 0; j < D; ++j) {
      const int4 dv = dev((uint32_t)j);
      const int32_t pk = dv.w + (weight ? *reinterpret_cast<const int32_t*>(ws_base + (uint32_t)j * pitch) : 0);   // the weights are resident from the start (Eq. 16)
      if (pk > cap[j]) st |= PE_STATUS_MEM_EXCEEDED;
      if (cand) {
        if (out.busy) out.busy[(size_t)j * (size_t)K + cc] = S16 ? (int32_t)((uint32_t)dv.y >> jb) : dv.y;
        if (out.peak_mem) out.peak_mem[(size_t)j * (size_t)K + cc] = pk;
      }
    }
    if (cand) {
      if (out.makespan) out.makespan[cc] = (int32_t)(z >> jb);
      if (out.status) out.status[cc] = st;
    }
  }
}

}  // namespace pe
