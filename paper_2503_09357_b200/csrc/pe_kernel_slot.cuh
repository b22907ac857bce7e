// One lane per candidate over the slot encoding: graphs through which only few results are alive at a time.
//
// Operators share state words ("slots").  Operator s takes over the slot of operator p when every successor of p is s or
// an ancestor of s: in any topological order all readers of p's end time are then through when s is scheduled.  The
// assignment of slots depends on the graph alone (made once in pe_graph_create), and a pipeline or a layered model graph
// needs few of them: 24 for the 1536 operators of the multi-modal graph.  So the per-candidate state shrinks from 4 bytes an
// operator to a few hundred bytes, and an SM holds hundreds of candidates instead of 14 to 60.
//
// The machine of an operator has no place in such a state, so the batch goes through two kernels:
//   pe_slot_gather_kernel   a block per tile of candidates, machine ids by operator in shared memory.  Nothing in it is
//                           serial: it looks up the machine of every position and sums the busy time and the resident
//                           weights of the machines.  Output: one word a position, operator | machine << 24, four positions
//                           of a candidate next to each other ([V / 4][K] of 16 bytes).
//   pe_eval_slot_kernel     the recurrence (Eqs. 3, 7-8, 11-13) and the memory levels (Eqs. 16-19), a lane per candidate.
//   pe_slot_times_kernel    start and finish by operator, where they are wanted: the recurrence leaves end time and
//                           machine by position, a tile is turned around in shared memory.
//
// Validity: a slot's operators are numbered in the order in which they hold it, and its word carries the number of the last
// one (its version).  Every reader compares the version that it finds with the one that it must find, and every operator
// reads the word of its own slot (as a predecessor's, or as one source more): a slot's operators are then executed one
// after the other, each once at most, and never before a predecessor.  V positions that pass are therefore a topological
// permutation, and every topological permutation passes.
// Graphs with many operators that nobody follows (OWN; random graphs, the bidirectional pipeline): such an operator needs no
// word, only a bit that says it has been executed.  That is the top bit of the version field of one of its predecessors, whose
// slot it leaves otherwise as it is; all operators then read the word of their own slot besides their sources'.
//
// State word: (time << vbits | version) << 8 | machine.
//
// What bounds them (counters of one launch, multi-modal graph V = 1536 K = 16384): the recurrence the chain of a step up to four
// warps on an SM (174 cycles a step, 58 instructions, 35 % of the issue slots, 43 % of the shared-memory pipe), then
// shared-memory wavefronts: 20.6 a step, 7 of them bank conflicts, mostly of the operator records.  The gather instructions
// and shared memory: 22 instructions and 8 wavefronts for 32 positions, 68 % of the pipe, 29 % of the DRAM rate (53 us for 25
// million positions).  Times by operator DRAM: 53 % of its rate (82 us).  The MoE graph takes 120 instructions and 30
// wavefronts a step, exclusive channels 79 and 22.5, marks (V = 1024 by position) 72 and 14.
// Measured on B200 (us, lane kernel with a word per operator, block of warps or global state before): multi-modal graph
// V = 1536 K = 65536 2304 -> 475 (gather 178, recurrence 274), K = 16384 594 -> 210, with durations by machine K = 32768 2320 ->
// 321, with exclusive channels K = 16384 1714 -> 467 (52, 413); MoE graph V = 2816 K = 16384 1850 -> 600, times by operator
// K = 16381 1918 -> 919 (118, 494, 305), with durations by machine K = 16384 11890 -> 748; V = 1024 D = 64 by position K = 2^19
// 7315 -> 5955 (980, 5090).
#pragma once
#include "pe_kernel_tile.cuh"
#include "pe_slot_shape.h"

namespace pe {

constexpr int kGatherThreads = 512;

__device__ __forceinline__ uint32_t min_u16x2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("min.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ uint32_t max_s16x2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("max.s16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ const uint8_t* row_at(const void* base, int row, uint32_t pitch) {   // one wide multiply-add
  return static_cast<const uint8_t*>(base) + (uint64_t)(uint32_t)row * pitch;
}
__device__ __forceinline__ uint8_t* row_at(void* base, int row, uint32_t pitch) {
  return static_cast<uint8_t*>(base) + (uint64_t)(uint32_t)row * pitch;
}

// C candidates a block.  Shared memory: machine ids by operator (u8 [V + 1][C], not BY_POS), busy times and weight sums ([D][C]
// each), status words.  Row V belongs to the entries that are no operator.
// A thread takes two candidates of a row where it looks up (a warp's accesses then spread over all banks) and four where
// it goes row by row.  VEC: rows can be read two order entries and four machine ids at a time.
template <int C, bool BY_POS, bool HET, bool VEC>
__global__ void __launch_bounds__(kGatherThreads, 2) pe_slot_gather_kernel(PeSlotView g, const uint8_t* __restrict__ sblob, int64_t K,
                                                                        int64_t n, const uint8_t* __restrict__ assign,
                                                                        const uint16_t* __restrict__ order, int32_t* __restrict__ busy_out,
                                                                        uint4* __restrict__ entries, int64_t pitch,
                                                                        uint32_t* __restrict__ status, int32_t* __restrict__ wsum_out) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  constexpr int T = kGatherThreads;
  const int V = g.V, D = g.D, tid = threadIdx.x;
  const uint32_t asg_bytes = BY_POS ? 0u : (uint32_t)(V + 1) * C;   // (a multiple of 8)
  uint8_t* asg = smem_raw;
  int32_t* busy = reinterpret_cast<int32_t*>(smem_raw + asg_bytes);
  int32_t* wsum = busy + D * C;
  uint32_t* flags = reinterpret_cast<uint32_t*>(wsum + (g.has_weight ? D * C : 0));   // [C], then: some machine id is out of range
  const uint16_t* dur = reinterpret_cast<const uint16_t*>(sblob + g.dur);
  const uint16_t* durm = reinterpret_cast<const uint16_t*>(sblob + g.durm);
  const int32_t* weight = g.has_weight ? reinterpret_cast<const int32_t*>(sblob + g.weight) : nullptr;
  const int64_t c0 = (int64_t)blockIdx.x * C;
  const uint32_t K1 = (uint32_t)K, K2 = (uint32_t)K * 2u;
  const uint32_t dmax = (uint32_t)(D - 1);
  // columns beyond the batch repeat its last candidate (the last full group of candidates with VEC) and are not written
  auto column = [&](int c, int group) -> size_t {
    const int64_t at = c0 + c;
    return (size_t)(VEC ? (at < n ? at : n - group) : (at < n ? at : n - 1));
  };
  auto busy_add = [&](uint32_t i, uint32_t j, int c, int32_t d) {   // d: the duration, without machines of their own
    atomicAdd(&busy[j * C + c], HET ? (int32_t)__ldg(durm + (size_t)i * D + j) >> g.vbits : d);
  };

  for (int q = tid; q < D * C * (g.has_weight ? 2 : 1); q += T) busy[q] = 0;
  if (!BY_POS && tid < C) asg[V * C + tid] = 0;
  for (int q = tid; q <= C; q += T) flags[q] = 0u;
  __syncthreads();

  constexpr int Q = C / 4, RQ = T / Q;   // groups of four, rows at once
  const int qc = 4 * (tid % Q), qr = tid / Q;
  if (!BY_POS) {   // machine ids by operator
    // a byte is >= D: bit 7 of (low seven bits + 128 - D) or of itself (D <= 128), of both with D - 128 beyond
    const uint32_t lift = (uint32_t)(D <= 128 ? 128 - D : 256 - D) * 0x01010101u;
    const uint8_t* asrc = assign + column(qc, 4);
    size_t off[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) off[q] = VEC ? 0 : column(qc + q, 4) - column(qc, 4);
    auto load_quad = [&](int i) -> uint32_t {
      const uint8_t* at = row_at(asrc, i, K1);
      if (VEC) return __ldg(reinterpret_cast<const uint32_t*>(at));
      return (uint32_t)__ldg(at) | (uint32_t)__ldg(at + off[1]) << 8 | (uint32_t)__ldg(at + off[2]) << 16 | (uint32_t)__ldg(at + off[3]) << 24;
    };
    constexpr int kBatch = 4;
    for (int b = qr; b < V; b += RQ * kBatch) {
      uint32_t x[kBatch], d[kBatch];
#pragma unroll
      for (int q = 0; q < kBatch; ++q) {
        const int i = min(b + q * RQ, V - 1);
        x[q] = load_quad(i);
        d[q] = HET ? 0u : (uint32_t)__ldg(dur + i);
      }
#pragma unroll
      for (int q = 0; q < kBatch; ++q) {
        const int i = b + q * RQ;
        if (i >= V) break;
        const uint32_t m = (x[q] & 0x7F7F7F7Fu) + lift;
        if ((D <= 128 ? (m | x[q]) : (m & x[q])) & 0x80808080u) {
          flags[C] = 1u;
          x[q] = __vminu4(x[q], dmax * 0x01010101u);
        }
        *reinterpret_cast<uint32_t*>(asg + i * C + qc) = x[q];
#pragma unroll
        for (int h = 0; h < 4; ++h) busy_add((uint32_t)i, (x[q] >> (8 * h)) & 0xFFu, qc + h, (int32_t)d[q]);
        if (weight)
#pragma unroll
          for (int h = 0; h < 4; ++h) atomicAdd(&wsum[((x[q] >> (8 * h)) & 0xFFu) * C + qc + h], __ldg(weight + i));
      }
    }
    __syncthreads();
  }

  const uint32_t vv = (uint32_t)V * 0x10001u;
  constexpr int H = C / 2, RH = T / H;   // pairs of a row, rows at once
  const int hc = 2 * (tid % H), hr = tid / H;
  const uint16_t* osrc = order + column(hc, 2);
  const size_t odd = VEC ? 1 : column(hc + 1, 2) - column(hc, 2);   // (second candidate of the pair, one element at a time)
  auto load_pair = [&](int k) -> uint32_t {   // order entries of two candidates, clamped to V
    const uint16_t* at = reinterpret_cast<const uint16_t*>(row_at(osrc, k, K2));
    const uint32_t x = VEC ? __ldg(reinterpret_cast<const uint32_t*>(at)) : ((uint32_t)__ldg(at) | (uint32_t)__ldg(at + odd) << 16);
    return min_u16x2(x, vv);
  };
  const bool have0 = c0 + hc < n, have1 = c0 + hc + 1 < n;
  const uint8_t* asrc = assign + column(hc, 2);
  {   // the words of the recurrence
    uint4* dst = entries + c0 + hc;
    const uint32_t pitch16 = (uint32_t)pitch * 16u;
    const int nq = (V + 3) >> 2, nfull = V >> 2;
    uint32_t most = 0;   // (halves: an entry that is no operator is V by now)
    auto emit = [&](int row, const uint32_t* o, const uint32_t* a) {
      uint32_t w0[4], w1[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t i0 = o[q] & 0xFFFFu, i1 = o[q] >> 16;
        asm("max.u16x2 %0, %0, %1;" : "+r"(most) : "r"(o[q]));
        uint32_t j0, j1;
        if (BY_POS) {
          const uint32_t r0 = a[q] & 0xFFu, r1 = a[q] >> 8;
          j0 = min(r0, dmax); j1 = min(r1, dmax);
          if (4 * row + q < V) {   // (an entry that is no operator consults no machine id)
            if (i0 < (uint32_t)V) {
              if (j0 != r0) atomicOr(&flags[hc], PE_STATUS_ASSIGN_RANGE);
              busy_add(i0, j0, hc, HET ? 0 : (int32_t)__ldg(dur + i0));
              if (weight) atomicAdd(&wsum[j0 * C + hc], __ldg(weight + i0));
            }
            if (i1 < (uint32_t)V) {
              if (j1 != r1) atomicOr(&flags[hc + 1], PE_STATUS_ASSIGN_RANGE);
              busy_add(i1, j1, hc + 1, HET ? 0 : (int32_t)__ldg(dur + i1));
              if (weight) atomicAdd(&wsum[j1 * C + hc + 1], __ldg(weight + i1));
            }
          }
        } else {
          j0 = asg[i0 * C + hc]; j1 = asg[i1 * C + hc + 1];
        }
        w0[q] = __byte_perm(o[q], j0, 0x4710);
        w1[q] = __byte_perm(o[q], j1, 0x4732);
      }
      uint4* at = reinterpret_cast<uint4*>(row_at(dst, row, pitch16));
      if (have0) at[0] = make_uint4(w0[0], w0[1], w0[2], w0[3]);
      if (have1) at[1] = make_uint4(w1[0], w1[1], w1[2], w1[3]);
    };
    auto load_a = [&](int k) -> uint32_t {
      return BY_POS ? (uint32_t)__ldg(row_at(asrc, k, K1)) | (uint32_t)__ldg(row_at(asrc, k, K1) + odd) << 8 : 0u;
    };
    int row = hr;
    for (; row + RH < nfull; row += 2 * RH) {
      uint32_t o[8], a[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int k = 4 * (row + (q >> 2) * RH) + (q & 3);
        o[q] = load_pair(k);
        a[q] = load_a(k);
      }
      emit(row, o, a);
      emit(row + RH, o + 4, a + 4);
    }
    for (; row < nq; row += RH) {
      uint32_t o[4], a[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int k = min(4 * row + q, V - 1);
        o[q] = load_pair(k);
        a[q] = load_a(k);
      }
      emit(row, o, a);
    }
    if ((most & 0xFFFFu) == (uint32_t)V) atomicOr(&flags[hc], PE_STATUS_ORDER_INVALID);
    if (most >> 16 == (uint32_t)V) atomicOr(&flags[hc + 1], PE_STATUS_ORDER_INVALID);
  }
  if (!BY_POS && flags[C] != 0u)   // some machine id was clamped: due where its operator is consulted
    for (int k = hr; k < V; k += RH) {
      const uint32_t o = load_pair(k), i0 = o & 0xFFFFu, i1 = o >> 16;
      if (i0 < (uint32_t)V && (uint32_t)*row_at(asrc, (int)i0, K1) > dmax) atomicOr(&flags[hc], PE_STATUS_ASSIGN_RANGE);
      if (i1 < (uint32_t)V && (uint32_t)*(row_at(asrc, (int)i1, K1) + odd) > dmax) atomicOr(&flags[hc + 1], PE_STATUS_ASSIGN_RANGE);
    }
  __syncthreads();
  for (int q = tid; q < C; q += T)
    if (c0 + q < n) status[c0 + q] = flags[q];
  for (int q = tid; q < D * C; q += T) {
    const int j = q / C, c = q % C;
    if (c0 + c >= n) continue;
    if (busy_out) busy_out[(size_t)j * (size_t)K + (size_t)(c0 + c)] = busy[q];
    if (weight) wsum_out[(size_t)j * (size_t)pitch + (size_t)(c0 + c)] = wsum[q];
  }
}

// Start and finish by operator.  words: state words by position, [V][pitch].
template <int C, bool HET>
__global__ void __launch_bounds__(kGatherThreads, 2) pe_slot_times_kernel(PeSlotView g, const uint8_t* __restrict__ sblob, int64_t K,
                                                                       int64_t n, const uint4* __restrict__ entries,
                                                                       const uint32_t* __restrict__ words, int64_t pitch,
                                                                       int32_t* __restrict__ start, int32_t* __restrict__ finish) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  constexpr int T = kGatherThreads, R = T / C;
  uint32_t* tile = reinterpret_cast<uint32_t*>(smem_raw);   // [V + 1][C]
  const int V = g.V, D = g.D;
  const int tid = threadIdx.x, c = tid % C, r0 = tid / C;
  const uint16_t* dur = reinterpret_cast<const uint16_t*>(sblob + g.dur);
  const uint16_t* durm = reinterpret_cast<const uint16_t*>(sblob + g.durm);
  const int64_t c0 = (int64_t)blockIdx.x * C;
  const bool cand = c0 + c < n;
  const size_t cc = (size_t)(cand ? c0 + c : n - 1);
  const int nq = (V + 3) >> 2;
  const uint32_t pitch4 = (uint32_t)pitch * 4u, K4 = (uint32_t)K * 4u;
  for (int b = r0; b < nq; b += R * 2) {
    uint4 e[2];
    uint32_t w[8];
#pragma unroll
    for (int h = 0; h < 2; ++h)
      e[h] = b + h * R < nq ? __ldg(reinterpret_cast<const uint4*>(row_at(entries + cc, b + h * R, pitch4 * 4u))) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int k = 4 * (b + (q >> 2) * R) + (q & 3);
      w[q] = k < V ? __ldg(reinterpret_cast<const uint32_t*>(row_at(words + cc, k, pitch4))) : 0u;
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int k = 4 * (b + (q >> 2) * R) + (q & 3);
      const uint4& v = e[q >> 2];
      const uint32_t x = (q & 3) == 0 ? v.x : ((q & 3) == 1 ? v.y : ((q & 3) == 2 ? v.z : v.w));
      if (k < V) tile[(x & 0xFFFFu) * C + c] = w[q];
    }
  }
  __syncthreads();
  if (!cand) return;
#pragma unroll 4
  for (int i = r0; i < V; i += R) {
    const uint32_t w = tile[i * C + c];
    const int32_t fin = (int32_t)(w >> (8 + g.vbits));
    const int32_t d = HET ? (int32_t)__ldg(durm + (size_t)i * D + min(w & 0xFFu, (uint32_t)(D - 1))) >> g.vbits : (int32_t)__ldg(dur + i);
    *reinterpret_cast<int32_t*>(row_at(start + cc, i, K4)) = fin - d;
    *reinterpret_cast<int32_t*>(row_at(finish + cc, i, K4)) = fin;
  }
}

// MODE of the recurrence
constexpr int kSlotPlain = 0;
constexpr int kSlotExcl = 1;     // PE_COMM_EXCLUSIVE: the end of the last transfer per channel, [machine pair][P], 32 bits
constexpr int kSlotExcl16 = 2;   // the same in 16 bits (time bounds below 2^16)
constexpr int kSlotHet = 3;      // durations by machine

// A step: machine record {end of the machine's last operator (packed), level << 16 | peak} and the words of the sources come
// from shared memory, everything else of the position was fetched during the step before.  (With the busy time in the record,
// 12 bytes, the gather is free of atomics, but fewer candidates fit: multi-modal graph K = 65536 474 -> 525 us, MoE graph
// K = 16381 922 -> 903.)
// CLS: 0 = one link class, every pair connected; 1 = class table; 2 = two classes, every pair connected, at most 32 machines.
// EDGES: no operator has more sources (1 to 3 with one class, 2 otherwise), all inline; 8 = inline ones, then six places of
// the list; 0 = inline ones, then the list.
// TIMES: 0 = none, 1 = by position, 2 = words for pe_slot_times_kernel.
// OWN: see above (one link class, EDGES 1 to 3, no channels).
template <int CLS, int EDGES, int TIMES, int MODE, bool OWN>
__global__ void __launch_bounds__(32 * kSlotWarps, 1) pe_eval_slot_kernel(PeSlotView g, const uint8_t* __restrict__ blob, int64_t K,
                                                                       int64_t n, const uint4* __restrict__ entries, int64_t pitch_e,
                                                                       const uint32_t* __restrict__ status, const int32_t* __restrict__ wsum,
                                                                       uint32_t* __restrict__ words, pe_outputs out, int* err, SlotShape sh) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  constexpr uint32_t FULL = 0xFFFFFFFFu;
  constexpr bool EXCL = MODE == kSlotExcl || MODE == kSlotExcl16, CH16 = MODE == kSlotExcl16, HET = MODE == kSlotHet;
  constexpr bool LIST = EDGES == 0 || EDGES == 8;
  constexpr int NIN = CLS == 0 ? (LIST ? 3 : EDGES) : 2;
  const int V = g.V, D = g.D;
  const int lane = threadIdx.x & 31;
  const int warp = __shfl_sync(FULL, (int)(threadIdx.x >> 5), 0);
  const int nwarps = blockDim.x >> 5;
  const int P = sh.lanes;
  {
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw + g.bytes);
    if (!stage_blob(smem_raw, blob, g.bytes, bar, err)) return;
  }
  const int32_t* cap = reinterpret_cast<const int32_t*>(smem_raw + g.cap);
  const uint32_t tshift = 8u + (uint32_t)g.vbits, tmask = ~0u << tshift, mark = 1u << (tshift - 1u);   // time field of a packed word, top bit of its version
  const uint32_t pitch = (uint32_t)P * 4u, dpitch = (uint32_t)P * 8u;
  const int ml = lane < P ? lane : P - 1;
  const bool mine = lane < P;
  const uint32_t dmax = (uint32_t)(D - 1), nslots = (uint32_t)g.nslots;
  const uint32_t smem_a = smem_u32(smem_raw);
  const uint32_t rec_a = smem_a + g.ops, cls_a = smem_a + g.cls, row_a = smem_a + g.cls_row, durm_a = smem_a + g.durm;
  const uint32_t list_a = smem_a + g.list, at_a = smem_a + g.list_at;
  const uint32_t st_a = smem_a + sh.off_state + (uint32_t)warp * sh.state_bytes + (uint32_t)ml * 4u;
  const uint32_t dv_a = smem_a + sh.off_dev + (uint32_t)warp * sh.dev_bytes + (uint32_t)ml * 8u;
  const uint32_t ch_a = smem_a + sh.off_chan + (uint32_t)warp * sh.chan_bytes + (uint32_t)ml * (CH16 ? 2u : 4u);
  const uint32_t chpitch = (uint32_t)P * (CH16 ? 2u : 4u);
  const uint32_t rpitch = (uint32_t)P * 16u, ring_a = smem_a + sh.off_ring + (uint32_t)warp * (kSlotQuads * rpitch) + (uint32_t)ml * 16u;
  const uint32_t K4 = (uint32_t)K * 4u, P4 = (uint32_t)pitch_e * 4u, row_e = (uint32_t)pitch_e * 16u;
  const int nq = (V + 3) >> 2;

  for (int64_t tile = (int64_t)warp * gridDim.x + blockIdx.x; tile < sh.tiles; tile += (int64_t)nwarps * gridDim.x) {
    const int64_t c0 = tile * P;
    const int in_tile = (int)(n - c0 < P ? n - c0 : P);
    const bool cand = lane < in_tile;
    const size_t cc = (size_t)c0 + (size_t)(lane < in_tile ? lane : in_tile - 1);
    const uint8_t* ent_b = reinterpret_cast<const uint8_t*>(entries) + cc * 16;
    // The words of a block of positions are brought to shared memory by asynchronous copies, each lane its own, while the
    // block before is worked on.  (Loads into registers share a scoreboard with the step's shared-memory loads: every
    // block then waited for DRAM.  Multi-modal graph K = 8192 158 -> 140 us when this was made.)
    uint4 cur[kSlotQuads];
    auto request = [&](int q0) {
#pragma unroll
      for (int q = 0; q < kSlotQuads; ++q)
        if (q0 + q < nq) cp_async16(ring_a + (uint32_t)q * rpitch, ent_b + (uint64_t)(uint32_t)q * row_e);
      ent_b += (uint64_t)kSlotQuads * row_e;
    };
    auto arrive = [&]() {
      cp_async_wait_all();
#pragma unroll
      for (int q = 0; q < kSlotQuads; ++q) cur[q] = lds128(ring_a + (uint32_t)q * rpitch);
    };
    __syncwarp();
    if (mine) {
      request(0);
      for (uint32_t q = 0; q < nslots + 1u; ++q) sts_state<false>(st_a + q * pitch, 0u);
      // (row nslots + 1 is only met by candidates that the gather has flagged: whatever it holds changes nothing.  Clearing it
      // too cost the form with marks and times by operator 2 %, 84.7 -> 86.2 us at V = 484 K = 16384.)
      for (int j = 0; j < D; ++j) sts64(dv_a + (uint32_t)j * dpitch, make_uint2(0u, 0u));
      if (EXCL)
        for (int q = 0; q < D * D; ++q) sts_state<CH16>(ch_a + (uint32_t)q * chpitch, 0u);
      arrive();
    }
    __syncwarp();

    uint32_t st = 0, bad = 0, marked = 0;   // bad: differences between versions found and expected, among other bits
    uint8_t* start_b = TIMES == 1 ? reinterpret_cast<uint8_t*>(out.start + cc) : reinterpret_cast<uint8_t*>(words + cc);
    uint8_t* finish_b = TIMES == 1 ? reinterpret_cast<uint8_t*>(out.finish + cc) : nullptr;
    uint32_t ent = mine ? cur[0].x : 0u;
    uint4 rec = lds128(rec_a + (ent & 0xFFFFu) * 16u);
    uint32_t dur_het = HET ? lds16(durm_a + ((ent & 0xFFFFu) * (uint32_t)D + (ent >> 24)) * 2u) : 0u;

    auto step = [&](const uint32_t ent_n) __attribute__((always_inline)) {
      const uint4 r4 = rec;
      const uint32_t j = ent >> 24;
      uint32_t p[NIN], w[NIN];
      if (CLS == 0) {
        p[0] = r4.y & 0xFFFu;
        if (NIN > 1) p[NIN > 1 ? 1 : 0] = r4.z & 0xFFFu;
        if (NIN > 2) p[NIN - 1] = LIST && (r4.z & 0x1000u) ? nslots : r4.w & 0xFFFu;
      } else {
        p[0] = r4.y & 0xFFFu;
        p[NIN - 1] = (r4.y >> 16) & 0xFFFu;
      }
#pragma unroll
      for (int q = 0; q < NIN; ++q) w[q] = lds32(st_a + p[q] * pitch);
      const uint32_t own_a = st_a + (((r4.x >> 16) & 0xFFu) | ((r4.y >> 4) & 0xF00u)) * pitch;
      const uint32_t w_own = OWN ? lds32(own_a) : 0u;
      const uint2 dv = lds64(dv_a + j * dpitch);
      uint32_t crow = 0;
      if (CLS == 2) crow = lds32(row_a + j * 4u);
      const uint4 rec_n = lds128(rec_a + (ent_n & 0xFFFFu) * 16u);
      uint32_t dur_n = 0;
      if (HET) dur_n = lds16(durm_a + ((ent_n & 0xFFFFu) * (uint32_t)D + (ent_n >> 24)) * 2u);

      auto pick = [&](uint32_t dd, uint32_t hi) -> uint32_t { return hi ? __byte_perm(dd, 0u, 0x4324) : __byte_perm(dd, 0u, 0x4104); };
      // One source: its packed end time plus the delay that applies (Eqs. 11-13).  The version that comes with the delay
      // meets the word's: both are below half of their field, so their sum stays out of the time.
      auto source = [&](uint32_t pp, uint32_t ww, uint32_t dd, bool real) __attribute__((always_inline)) -> uint32_t {
        const bool same = ((ww ^ j) & 0xFFu) == 0u;
        uint32_t d;
        bool channel = true;
        if (CLS == 0) {
          d = pick(dd, 1u);
          bad |= ww ^ d;
        } else if (CLS == 2) {
          d = pick(dd, __funnelshift_r(crow, crow, ww) & 1u);   // (shift amount modulo 32: the machine)
          bad |= ww ^ d;
        } else {
          const uint32_t cl = lds8(cls_a + min(ww & 0xFFu, dmax) * (uint32_t)D + j);
          d = pick(dd, cl == 1u ? 1u : 0u);
          bad |= ww ^ d;
          if (cl == 0xFFu) {
            d = 0u;
            channel = false;
            if (!same && pp != nslots && real) st |= PE_STATUS_NO_CHANNEL;
          }
        }
        if (EXCL) {
          // the transfer starts when its source has ended (Eq. 13) and the channel is free (Eq. 14), lasts D^c (Eq. 11).
          // Sources that need no channel take the word behind the last one: 32 candidates would take both sides of a branch.
          const bool moves = !same && pp != nslots && channel && real;
          const uint32_t ch = ch_a + (moves ? (ww & 0xFFu) * (uint32_t)D + j : (uint32_t)(D * D)) * chpitch;
          uint32_t t_end;
          if (CH16) {
            t_end = max(ww >> tshift, lds16(ch)) + (d >> tshift);
            sts_state<true>(ch, t_end);
            t_end <<= tshift;
          } else {
            t_end = max(ww & tmask, lds32(ch)) + (d & tmask);
            sts_state<false>(ch, t_end);
          }
          return moves ? t_end : ww;
        }
        return ww + (same ? 0u : d);
      };
      uint32_t r = dv.x;
      if (CLS == 0) {
        const bool first = (EXCL || CLS == 1) ? !(r4.z & 0x2000u) : true;
        r = max(r, source(p[0], w[0], r4.y, first));
        if (NIN > 1) r = max(r, source(p[NIN > 1 ? 1 : 0], w[NIN > 1 ? 1 : 0], r4.z, true));
        if (NIN > 2 && !(LIST && (r4.z & 0x1000u))) r = max(r, source(p[NIN - 1], w[NIN - 1], r4.w, true));
        if (LIST && (r4.z & 0x1000u)) {   // w: place of source 2 in the list
          uint32_t at = list_a + r4.w * 4u;
          if (EDGES == 8) {
            const uint4 a = lds128(at), b = lds128(at + 16u);
            const uint32_t ed[6] = {a.x, a.y, a.z, a.w, b.x, b.y};
            uint32_t lw[6];
#pragma unroll
            for (int q = 0; q < 6; ++q) lw[q] = lds32(st_a + (ed[q] & 0xFFFu) * pitch);
#pragma unroll
            for (int q = 0; q < 6; ++q) r = max(r, source(ed[q] & 0xFFFu, lw[q], ed[q], true));
          } else {
            uint32_t ed;
            do {   // up to the marked one
              ed = lds32(at);
              r = max(r, source(ed & 0xFFFu, lds32(st_a + (ed & 0xFFFu) * pitch), ed, true));
              at += 4u;
            } while (!(ed & 0x1000u));
          }
        }
      } else {
        const bool first = (EXCL || CLS == 1) ? !(r4.y & 0x20000000u) : true;
        r = max(r, source(p[0], w[0], r4.z, first));
        r = max(r, source(p[NIN - 1], w[NIN - 1], r4.w, true));
        if (LIST && (r4.y & 0x10000000u)) {
          uint32_t at = list_a + lds32(at_a + (ent & 0xFFFFu) * 4u) * 8u;
          if (EDGES == 8) {
            const uint4 a = lds128(at), b = lds128(at + 16u), c = lds128(at + 32u);
            const uint32_t es[6] = {a.x, a.z, b.x, b.z, c.x, c.z}, ed[6] = {a.y, a.w, b.y, b.w, c.y, c.w};
            uint32_t lw[6];
#pragma unroll
            for (int q = 0; q < 6; ++q) lw[q] = lds32(st_a + (es[q] & 0xFFFu) * pitch);
#pragma unroll
            for (int q = 0; q < 6; ++q) r = max(r, source(es[q] & 0xFFFu, lw[q], ed[q], true));
          } else {
            uint2 ed;
            do {
              ed = lds64(at);
              r = max(r, source(ed.x & 0xFFFu, lds32(st_a + (ed.x & 0xFFFu) * pitch), ed.y, true));
              at += 8u;
            } while (!(ed.x & 0x1000u));
          }
        }
      }
      const uint32_t durj = __byte_perm(r4.x, j, 0x5104);   // D^o, the own version and the machine (Eq. 3)
      const uint32_t rt = r & tmask;
      const uint32_t e = HET ? rt + durj + (dur_het << 8) : rt + durj;
      // + A_i (byte 3 of the record) on the level; the peak follows it (Eqs. 17-19)
      const uint32_t lv = dv.y + ((uint32_t)__dp4a((int32_t)r4.x, 0x01000000, 0) << 16);
      const uint32_t lp = max_s16x2(lv, __byte_perm(lv, 0u, 0x3232));
      if (OWN) {
        const bool last = (durj & mark) != 0u;   // nobody follows it
        if (last) marked |= w_own;
        else bad |= (w_own + 0x100u) ^ durj;
        sts_state<false>(own_a, last ? w_own | mark : e);
      } else {
        sts_state<false>(own_a, e);
      }
      sts64(dv_a + j * dpitch, make_uint2(e, lp));
      if (TIMES == 1) {
        *reinterpret_cast<int32_t*>(start_b) = (int32_t)(rt >> tshift);
        *reinterpret_cast<int32_t*>(finish_b) = (int32_t)(e >> tshift);
        start_b += K4;
        finish_b += K4;
      }
      if (TIMES == 2) {
        *reinterpret_cast<uint32_t*>(start_b) = e;
        start_b += P4;
      }
      ent = ent_n;
      rec = rec_n;
      dur_het = dur_n;
    };

    // (lanes beyond the tile would write the last lane's words: they stay out)
    constexpr int kStep = 4 * kSlotQuads;
    int kb = mine ? 0 : V;
    for (; kb + kStep <= V; kb += kStep) {
      request((kb >> 2) + kSlotQuads);
#pragma unroll
      for (int q = 0; q < kSlotQuads; ++q) {
        step(cur[q].y);
        step(cur[q].z);
        step(cur[q].w);
        if (q + 1 < kSlotQuads) step(cur[(q + 1) % kSlotQuads].x);
      }
      arrive();   // (what arrives behind the last position is not used)
      step(kb + kStep < V ? cur[0].x : 0u);
    }
    for (int k = kb; k < V; ++k) {   // the last positions, word by word
      const uint32_t at = (uint32_t)(k + 1 - kb);
      step(k + 1 < V ? lds32(ring_a + (at >> 2) * rpitch + (at & 3u) * 4u) : 0u);
    }
    __syncwarp();

    if ((bad & (mark - 0x100u)) | (marked & mark)) st |= PE_STATUS_ORDER_INVALID;
    uint32_t z = 0;
    st |= status[cc];
    for (int j = 0; j < D; ++j) {
      const uint2 dv = lds64(dv_a + (uint32_t)j * dpitch);
      z = max(z, dv.x);
      const int32_t pk = (int32_t)(int16_t)(dv.y & 0xFFFFu) + (wsum ? wsum[(size_t)j * (size_t)pitch_e + cc] : 0);   // the weights are resident from the start (Eq. 16)
      if (pk > cap[j]) st |= PE_STATUS_MEM_EXCEEDED;
      if (cand && out.peak_mem) out.peak_mem[(size_t)j * (size_t)K + cc] = pk;
    }
    if (cand) {
      if (out.makespan) out.makespan[cc] = (int32_t)(z >> tshift);
      if (out.status) out.status[cc] = st;
    }
  }
}

}  // namespace pe
