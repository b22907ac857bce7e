// pe_decode_priority: priority-list decoding, the step in front of pe_eval_batch.
//
// The paper prints no decoder (Section IV mentions dispatch rules only as the inspiration of its
// coarsening heuristic); the rule implemented here is this library's choice: a candidate ranks the operators through a list (list[r] =
// the operator of rank r; any permutation of I), and the priority order pi is built position by
// position: among the operators not yet placed whose predecessors in B have all been placed, the
// one of smallest rank comes next (Kahn's algorithm with the ranks as priorities).  The result is
// a topological order of G_m, i.e. a valid `order` argument of pe_eval_batch.
//
// The set of available operators is kept by rank.  Kernels:
//
// Warp per candidate (pe_decode_warp_kernel; per-operator state on chip).  Placing an operator is a chain of
// dependent steps (smallest rank -> operator -> successors -> their counts -> new ranks), so the work is spread
// over the lanes only where that shortens the chain:
//   word[i]   shared memory: rank of operator i (bits 0..15) | predecessors still missing (bits 16..31)
//   bitmap    shared memory: available operators of rank >= T
//   pool      registers: every available operator of rank < T, one per lane as rank << 16 | operator
// The smallest available rank is then one warp-wide minimum over the pool; an operator's successors are handled by
// the lanes whose pool place is free, so a released operator of rank < T stays where it was found, one of rank >= T
// sets its bit.  When the pool is empty the next bitmap words that together hold up to kFill operators are loaded into
// it and T moves behind those words; all words below T stay empty, so the scan over the bitmap is monotone.  If more
// operators are released than the pool has places, the pool goes back to the bitmap (T = 0) and fills again.
// What bounds it: instruction issue (52 warp instructions a placement, 85 % of the issue slots used at V = 480) while
// many warps fit, the chain (~270 cycles a placement with the records on chip) when few do.  Measured (before: a
// thread per candidate, state in shared memory up to V ~ 1100, else in the workspace): V = 480, K = 65536 2.21 -> 1.65
// ms, K = 1024 318 -> 78 us; V = 1536, K = 8192 3.14 -> 0.83 ms; V = 2816, K = 8192 9.97 -> 2.8 ms; V = 4096, K = 8192
// 27.5 -> 5.9 ms; V = 16384, K = 2048 125 -> 23.5 ms.  Candidate-major copies of list and order, and records brought
// to the pool's places by asynchronous copies, were measured and changed nothing or cost up to 15 %.
//
// Lane per candidate (pe_decode_lane_kernel; V <= 256, large batches).  The set of available operators is a bitmap
// with one summary word in a register; 3.1 bytes of state per operator (rank and missing predecessors in 16 bits, the
// list in 8) let up to ~1000 candidates share an SM and hide the chain of a placement, bitmap -> list -> successor
// list -> counts, about five shared-memory round trips.
//
// Lane per candidate with a pool (pe_decode_pool_kernel, see there): graphs that a few chains of operators cover.
//
// Thread per candidate (pe_decode_kernel; for graphs whose per-candidate state does not fit on chip, V above
// ~55000, or on request).  The bitmap has two summary levels above it (one bit per 32-bit word of the level below;
// the top level is a 64-bit register, which is why V <= 65536): "take the smallest" is three find-first-set steps.
// Words and bitmaps are in the caller's workspace in tiles of 32 candidates, [tile][row][32]; the list is read back
// from the input when a rank is taken, the successor lists through the cache.
#include <algorithm>
#include <atomic>
#include <climits>

#include "pe_device.cuh"
#include "pe_graph.h"
#include "pe_launch.h"
#include "pe_smem.cuh"

namespace pe {

extern std::atomic<int64_t> g_decode_launches;
std::atomic<int64_t> g_decode_launches{0};

struct FwdPtrs {
  const uint32_t* ptr;
  const uint16_t* succ;
  const uint8_t* indeg;
};

__device__ __forceinline__ FwdPtrs fwd_ptrs(const uint8_t* base, const PeFwdView& f) {
  FwdPtrs p;
  p.ptr = reinterpret_cast<const uint32_t*>(base + f.ptr);
  p.succ = reinterpret_cast<const uint16_t*>(base + f.succ);
  p.indeg = base + f.indeg;
  return p;
}

constexpr uint32_t kSeen = 0x80000000u;
constexpr uint32_t kFill = 16;              // operators that an empty pool is filled with: as many places stay free
constexpr size_t kDecodeRecBytes = 32768;   // operator records up to this size are kept in shared memory
constexpr int kListAhead = 8;  // rows of the list requested ahead of the one being placed

__global__ void __launch_bounds__(256) pe_decode_kernel(PeFwdView f, const uint8_t* __restrict__ fblob, int64_t K,
                                                        const uint16_t* __restrict__ list, uint16_t* __restrict__ order,
                                                        uint32_t* __restrict__ status, uint32_t* __restrict__ gstate) {
  const int T = blockDim.x;
  const int t = threadIdx.x;
  const int V = f.V;
  const FwdPtrs fp = fwd_ptrs(fblob, f);
  const int64_t c = (int64_t)blockIdx.x * T + t;
  if (c >= K) return;
  const size_t Ks = (size_t)K;
  const int n0 = (V + 31) >> 5, n1 = (n0 + 31) >> 5;
  // row r of this candidate's state is st[r * pitch]
  uint32_t* st = gstate + (size_t)(c >> 5) * (size_t)(V + n0 + n1) * 32 + (c & 31);
  constexpr uint32_t pitch = 32u;
  uint32_t* word = st;
  uint32_t* L0 = st + (size_t)V * pitch;
  uint32_t* L1 = L0 + (size_t)n0 * pitch;
  uint64_t L2 = 0;

  auto add = [&](uint32_t r) {   // rank r becomes available
    uint32_t* p0 = L0 + (r >> 5) * pitch;
    const uint32_t w0 = *p0;
    *p0 = w0 | (1u << (r & 31u));
    if (w0 == 0u) {              // the word was empty: the levels above learn of it
      L1[(r >> 10) * pitch] |= 1u << ((r >> 5) & 31u);
      L2 |= 1ull << (r >> 10);
    }
  };

  for (int i = 0; i < V; ++i) word[(uint32_t)i * pitch] = (uint32_t)fp.indeg[i] << 16;
  for (int q = 0; q < n0 + n1; ++q) L0[(uint32_t)q * pitch] = 0u;

  // the list: rank and "seen" into the operators' words, operators without predecessors become available
  const uint16_t* list_col = list + c;
  bool bad = false;
  {
    uint32_t ring[kListAhead];
#pragma unroll
    for (int u = 0; u < kListAhead; ++u) ring[u] = (uint32_t)list_col[(size_t)min(u, V - 1) * Ks];
    for (int r0 = 0; r0 < V; r0 += kListAhead) {
      uint32_t cur[kListAhead];
#pragma unroll
      for (int u = 0; u < kListAhead; ++u) {
        cur[u] = ring[u];
        ring[u] = (uint32_t)list_col[(size_t)min(r0 + kListAhead + u, V - 1) * Ks];
      }
#pragma unroll
      for (int u = 0; u < kListAhead; ++u) {
        const int r = r0 + u;
        if (r < V) {
          const uint32_t i = cur[u];
          if (i >= (uint32_t)V) {
            bad = true;
          } else {
            const uint32_t w = word[i * pitch];
            if (w & kSeen) {
              bad = true;            // the operator is in the list twice
            } else {
              word[i * pitch] = w | kSeen | (uint32_t)r;
              if ((w >> 16) == 0u) add((uint32_t)r);
            }
          }
        }
      }
    }
  }
  if (status) status[c] = bad ? (uint32_t)PE_STATUS_ORDER_INVALID : 0u;
  if (bad) return;   // not a permutation: the order of this candidate stays unwritten

  // Main loop.  Every iteration hands one successor of the operator placed last its "one predecessor fewer"
  // and, once that operator's successor list is used up, places the next operator.  All candidates share the
  // graph, so every lane needs the same number of successor steps and placements in total; spreading them
  // over uniform iterations keeps the lanes of a warp busy where a loop over each operator's successors
  // would make the whole warp wait for the lane that drew the operator with the most successors.
  uint16_t* order_col = order + c;
  uint32_t e = 0, e_end = 0;
  int k = 0;
  for (int it = 0; it < 2 * V + f.E + 2; ++it) {   // (bound: at most V placements and E successor steps)
    if (e < e_end) {
      const uint32_t s = fp.succ[e++];
      const uint32_t w = word[s * pitch] - (1u << 16);
      word[s * pitch] = w;
      if (((w >> 16) & 0xFFu) == 0u) add(w & 0xFFFFu);
    }
    if (e == e_end) {
      if (k == V || L2 == 0) break;   // all placed (L2 == 0 earlier cannot happen for a permutation over a DAG)
      // the smallest available rank: first set bit of each level, top down
      const uint32_t b2 = (uint32_t)__ffsll((long long)L2) - 1u;
      uint32_t w1 = L1[b2 * pitch];
      if (w1 == 0u) break;   // (a summary bit without anything below it: cannot happen either)
      const uint32_t b1 = (uint32_t)__ffs((int)w1) - 1u;
      const uint32_t i0 = b2 * 32u + b1;
      uint32_t w0 = L0[i0 * pitch];
      if (w0 == 0u) break;
      const uint32_t b0 = (uint32_t)__ffs((int)w0) - 1u;
      const uint32_t r = i0 * 32u + b0;
      w0 &= ~(1u << b0);
      L0[i0 * pitch] = w0;
      if (w0 == 0u) {
        w1 &= ~(1u << b1);
        L1[b2 * pitch] = w1;
        if (w1 == 0u) L2 &= ~(1ull << b2);
      }
      const uint32_t i = (uint32_t)list_col[(size_t)r * Ks];
      order_col[(size_t)k * Ks] = (uint16_t)i;
      ++k;
      e = fp.ptr[i];
      e_end = fp.ptr[i + 1];
    }
  }
}

constexpr uint32_t kNoKey = 0xFFFFFFFFu;   // an empty pool place (V <= 65535: no key equals it)

// REC_SMEM: the operator records are copied to shared memory in front of the warps' words.
template <bool REC_SMEM>
__global__ void __launch_bounds__(256) pe_decode_warp_kernel(PeFwdView f, const uint8_t* __restrict__ fblob, int64_t K,
                                                             const uint16_t* __restrict__ list, uint16_t* __restrict__ order,
                                                             uint32_t* __restrict__ status, uint32_t words) {
  extern __shared__ __align__(16) uint32_t smem_words[];
  constexpr uint32_t FULL = 0xFFFFFFFFu;
  constexpr uint32_t kOne = 1u << 16;   // one missing predecessor
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t c = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
  const int V = f.V;
  const uint32_t rb = f.rec_bytes, inl2 = f.rec_bytes - 4u;   // bytes of a record, of its inline successors
  const uint8_t* indeg = fblob + f.indeg;
  const uint8_t* rec_g = fblob + f.rec;
  const uint16_t* more = reinterpret_cast<const uint16_t*>(fblob + f.more);
  if (REC_SMEM) {
    uint4* copy = reinterpret_cast<uint4*>(smem_words);
    const int n16 = V * (int)(rb >> 4);
    for (int i = threadIdx.x; i < n16; i += blockDim.x) copy[i] = __ldg(reinterpret_cast<const uint4*>(rec_g) + i);
    __syncthreads();
  }
  if (c >= K) return;
  const uint32_t rec_a = smem_u32(smem_words);
  // word[V] is the operator that empty record places name: it misses more predecessors than there are placements, and
  // each placement takes off one at most
  uint32_t* word = smem_words + (REC_SMEM ? (size_t)V * (rb >> 2) : 0) + (size_t)warp * words;
  uint32_t* bitmap = word + V + 1;
  uint32_t* found = bitmap + ((V + 31) >> 5);   // ranks on their way from the bitmap to the pool
  const uint32_t word_a = smem_u32(word);
  const int nb = (V + 31) >> 5;
  const size_t row = (size_t)K;
  const uint16_t* list_c = list + c;
  uint16_t* order_c = order + c;
  const uint32_t lt_mask = (1u << lane) - 1u;

  for (int i = lane; i <= V; i += 32) word[i] = 0xFFFFFFFFu;
  __syncwarp();
  // ranks into the operators' words; operators without predecessors are available
  bool bad = false;
  constexpr int kBatch = 8;
  for (int b = 0; b < nb; b += kBatch) {
    uint32_t i[kBatch], m[kBatch];
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
      const int r = (b + q) * 32 + lane;
      i[q] = r < V ? (uint32_t)list_c[(size_t)r * row] : 0xFFFFFFFFu;
      bad = bad || (r < V && i[q] >= (uint32_t)V);
    }
#pragma unroll
    for (int q = 0; q < kBatch; ++q) m[q] = i[q] < (uint32_t)V ? (uint32_t)__ldg(indeg + i[q]) : 1u;
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
      if (i[q] < (uint32_t)V) word[i[q]] = m[q] * kOne | (uint32_t)((b + q) * 32 + lane);
      const uint32_t avail = __ballot_sync(FULL, m[q] == 0u);
      if (lane == 0 && b + q < nb) bitmap[b + q] = avail;
    }
  }
  __syncwarp();
  for (int i = lane; i < V; i += 32) bad = bad || word[i] == 0xFFFFFFFFu;   // an operator twice leaves another one out
  bad = __any_sync(FULL, bad);
  if (status && lane == 0) status[c] = bad ? (uint32_t)PE_STATUS_ORDER_INVALID : 0u;
  if (bad) return;   // not a permutation: the order of this candidate stays unwritten

  uint32_t hot = kNoKey;      // this lane's pool place
  uint32_t T = 0;             // ranks below T are in the pool, the others in the bitmap
  int scan = 0;               // bitmap words below are empty
  // one successor: one predecessor fewer; released (its word is its rank now), it takes this lane's place or its bit
  auto handle = [&](uint32_t s) {
    const uint32_t at = word_a + s * 4u;
    uint32_t w;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(w) : "r"(at));
    w -= kOne;
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(at), "r"(w) : "memory");
    if (w < T) hot = __byte_perm(w, s, 0x1054);
    if (w - T < kOne - T) atomicOr(&bitmap[w >> 5], 1u << (w & 31u));
  };
  // (every turn places an operator or fills an empty pool, which the next turn takes from: at most 2 V turns)
  while (true) {
    // free places and this lane's number among them (the place of the operator taken now counts from the next turn on)
    const uint32_t open = __ballot_sync(FULL, hot == kNoKey);
    const uint32_t key = __reduce_min_sync(FULL, hot);
    if (key == kNoKey) {      // the next words of the bitmap that hold up to kFill operators (or more in the first one)
      uint32_t total = 0;
      while (total == 0u && scan < nb) {
        uint32_t x = scan + lane < nb ? bitmap[scan + lane] : 0u;
        if (!__any_sync(FULL, x != 0u)) { scan += 32; continue; }
        const uint32_t cnt = (uint32_t)__popc(x);
        uint32_t incl = cnt;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const uint32_t o = __shfl_up_sync(FULL, incl, off);
          incl += lane >= off ? o : 0u;
        }
        const bool take = incl <= kFill || incl == cnt;   // a prefix of the words
        const int nw = __popc(__ballot_sync(FULL, take));
        total = __shfl_sync(FULL, incl, nw - 1);
        if (take && x != 0u) {
          bitmap[scan + lane] = 0u;
          for (uint32_t at = incl - cnt; x != 0u; x &= x - 1u) found[at++] = 32u * (uint32_t)(scan + lane) + (uint32_t)__ffs((int)x) - 1u;
        }
        scan = min(scan + nw, nb);
      }
      if (total == 0u) break;   // all placed
      T = 32u * (uint32_t)scan;
      __syncwarp();
      if ((uint32_t)lane < total) {
        const uint32_t r = found[lane];
        hot = (r << 16) | (uint32_t)list_c[(size_t)r * row];
      }
      __syncwarp();
      continue;
    }
    const uint32_t i = key & 0xFFFFu;
    const bool mine = hot == kNoKey;
    uint32_t t = mine ? (uint32_t)__popc(open & lt_mask) * 2u : inl2;
    t = min(t, inl2);
    uint32_t n, s;
    if (REC_SMEM) {
      const uint32_t at = rec_a + i * rb;
      uint16_t h, g;
      asm volatile("ld.shared.u16 %0, [%1];" : "=h"(h) : "r"(at));
      asm volatile("ld.shared.u16 %0, [%1];" : "=h"(g) : "r"(at + t + 2u));
      n = h; s = g;
    } else {
      const uint8_t* at = rec_g + i * rb;
      n = __ldg(reinterpret_cast<const uint16_t*>(at));
      s = __ldg(reinterpret_cast<const uint16_t*>(at + t + 2u));
    }
    if (lane == 0) *order_c = (uint16_t)i;
    order_c += row;
    if (hot == key) hot = kNoKey;
    if (n <= (uint32_t)__popc(open)) {   // (n is 64 in the record of an operator with a longer list)
      handle(s);
      __syncwarp();
      continue;
    }
    // an operator with a longer list, or fewer free places than successors
    const uint16_t* r8 = reinterpret_cast<const uint16_t*>(rec_g + (size_t)i * rb);
    const bool listed = n > 32u;
    const uint16_t* list_s = listed ? more + ((uint32_t)__ldg(r8 + 2) | (uint32_t)__ldg(r8 + 3) << 16) : r8 + 1;
    if (listed) n = __ldg(r8 + 1);
    for (uint32_t done = 0; done < n;) {
      uint32_t free_now = __ballot_sync(FULL, hot == kNoKey);
      if (free_now == 0u) {   // the pool is full: back to the bitmap with it
        const uint32_t r = hot >> 16;
        atomicOr(&bitmap[r >> 5], 1u << (r & 31u));
        hot = kNoKey;
        T = 0u;
        scan = 0;
        free_now = FULL;
        __syncwarp();
      }
      const uint32_t q = done + (uint32_t)__popc(free_now & lt_mask);
      if (hot == kNoKey && q < n) handle((uint32_t)__ldg(list_s + q));
      done += (uint32_t)__popc(free_now);
      __syncwarp();
    }
  }
}

// The block's threads keep word[i] (rank of operator i | missing predecessors << 8) and list[r] as [row][thread]; two
// (four) warps share the 32-bit words of a row, so that the lanes of a warp fall into different banks.
constexpr int kLaneThreads = 128;
__global__ void __launch_bounds__(kLaneThreads) pe_decode_lane_kernel(PeFwdView f, const uint8_t* __restrict__ fblob, int64_t K,
                                                                      const uint16_t* __restrict__ list,
                                                                      uint16_t* __restrict__ order, uint32_t* __restrict__ status) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  const int V = f.V, E = f.E, t = threadIdx.x;
  const FwdPtrs fp = fwd_ptrs(fblob, f);
  uint32_t* head = reinterpret_cast<uint32_t*>(smem_raw);   // first successor | how many << 16 | missing predecessors << 24
  uint32_t* bits = head + V;                                // [(V + 31) / 32][thread]
  const int nb = (V + 31) >> 5;
  uint16_t* words = reinterpret_cast<uint16_t*>(bits + nb * kLaneThreads);
  uint8_t* lists = reinterpret_cast<uint8_t*>(words + V * kLaneThreads);
  uint8_t* succ = lists + V * kLaneThreads;
  for (int i = t; i < V; i += kLaneThreads) {
    const uint32_t b = fp.ptr[i];
    head[i] = b | (fp.ptr[i + 1] - b) << 16 | (uint32_t)fp.indeg[i] << 24;   // (a predecessor list is at most 255 long)
  }
  for (int e = t; e < E; e += kLaneThreads) succ[e] = (uint8_t)fp.succ[e];
  __syncthreads();
  const int64_t c = (int64_t)blockIdx.x * kLaneThreads + t;
  if (c >= K) return;
  const size_t Ks = (size_t)K;
  uint16_t* word = words + 2 * (32 * (t >> 6) + (t & 31)) + ((t >> 5) & 1);
  uint8_t* lst = lists + 4 * (t & 31) + (t >> 5);
  uint32_t* bit = bits + t;
  uint32_t some = 0;   // bitmap words that are not empty
  auto add = [&](uint32_t r) {
    bit[(r >> 5) * kLaneThreads] |= 1u << (r & 31u);
    some |= 1u << (r >> 5);
  };
  for (int q = 0; q < nb; ++q) bit[q * kLaneThreads] = 0u;
  for (int i = 0; i < V; ++i) word[i * kLaneThreads] = 0xFFFFu;
  bool bad = false;
  const uint16_t* list_c = list + c;
  constexpr int kBatch = 16;
  for (int r0 = 0; r0 < V; r0 += kBatch) {
    uint32_t i[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) i[u] = (uint32_t)list_c[(size_t)min(r0 + u, V - 1) * Ks];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int r = r0 + u;
      if (r < V) {
        bad = bad || i[u] >= (uint32_t)V;
        const uint32_t op = min(i[u], (uint32_t)(V - 1));
        const uint32_t missing = head[op] >> 24;
        bad = bad || word[op * kLaneThreads] != 0xFFFFu;   // twice (0xFFFF is also what 255 missing at rank 255 make, but that is the last entry: nothing follows that could meet it)
        lst[r * kLaneThreads] = (uint8_t)op;
        word[op * kLaneThreads] = (uint16_t)(missing << 8 | (uint32_t)r);
        if (missing == 0u) add((uint32_t)r);
      }
    }
  }
  if (status) status[c] = bad ? (uint32_t)PE_STATUS_ORDER_INVALID : 0u;
  if (bad) return;   // not a permutation: the order of this candidate stays unwritten

  // Every iteration hands one successor of the operator placed last its "one predecessor fewer" and, once that
  // operator's list is used up, places the next one: all lanes need the same number of either in total.
  uint16_t* order_c = order + c;
  uint32_t e = 0, e_end = 0;
  int k = 0;
  for (int it = 0; it < V + E + 2; ++it) {   // (bound: V placements, E successor steps)
    if (e < e_end) {
      const uint32_t s = succ[e++];
      const uint32_t w = (uint32_t)word[s * kLaneThreads] - 0x100u;
      word[s * kLaneThreads] = (uint16_t)w;
      if ((w >> 8) == 0u) add(w & 0xFFu);
    }
    if (e == e_end) {
      if (k == V) break;
      if (some == 0u) break;   // (cannot happen for a permutation over a DAG)
      const uint32_t q = (uint32_t)__ffs((int)some) - 1u;
      const uint32_t x = bit[q * kLaneThreads];
      const uint32_t r = 32u * q + (uint32_t)__ffs((int)x) - 1u;
      bit[q * kLaneThreads] = x & (x - 1u);
      if ((x & (x - 1u)) == 0u) some &= some - 1u;
      const uint32_t i = lst[r * kLaneThreads];
      *order_c = (uint16_t)i;
      order_c += Ks;
      ++k;
      const uint32_t h = head[i];
      e = h & 0xFFFFu;
      e_end = e + ((h >> 16) & 0xFFu);
    }
  }
}

// Shape of a pe_decode_pool_kernel launch: warps take tiles of `lanes` candidates.
struct PoolShape {
  int lanes;
  int64_t tiles;
  uint32_t off_state;     // state of warp 0: pool, ranks, counts
  uint32_t state_bytes;   // per warp
  uint32_t off_rank, off_cnt;
};

// Lane per candidate with a pool (pe_decode_pool_kernel): graphs that at most 32 chains cover (two operators
// of a chain, one an ancestor of the other, are never available together).  The available operators stand in shared memory, [place / 4][lane][4], as rank << 17 |
// place << 12 | operator; a lane reads all places to find the smallest rank, three instructions for four places.
//   rank[i]   u16 [operator][lane]: rank of operator i
//   cnt[j]    u8 [join][lane]: predecessors still missing, less one, of the operators that have several; row num_joins
//             stands for all others (always 0), row num_joins + 1 takes what they write
// Every turn of the loop hands one successor of the operator placed last its "one predecessor fewer" and, once that
// operator's list is used up, places the next one.  A turn has no branch (32 candidates would take every side of each: a
// first version with them took 730 cycles a turn), and the pool is read while the successor's rank is on its way: what
// is released in this turn is compared with what was in the pool before.
// What bounds it: the chain operator -> record -> rank of its successor, two shared-memory round trips, with the few warps
// that fit (2 bytes an operator and candidate): 249 cycles a turn, set-up included, at V = 1536 K = 8192 (two warps on an SM, 109
// instructions and 38 shared-memory wavefronts a turn, 45 % of the issue slots of the schedulers that have a warp).  Measured
// (us, warp kernel or lane kernel with a bitmap before): multi-modal graph V = 1536 K = 8192 834 -> 199, K = 64 231 -> 192; MoE
// graph V = 2816 K = 8192 2785 -> 1258; pipeline V = 256 K = 16384 100 -> 41, V = 64 K = 1024 18 -> 14.
template <int QUADS>
__global__ void __launch_bounds__(512, 1) pe_decode_pool_kernel(PeFwdView f, const uint8_t* __restrict__ fblob, int64_t K,
                                                                const uint16_t* __restrict__ list, uint16_t* __restrict__ order,
                                                                uint32_t* __restrict__ status, PoolShape sh, int* err) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  const int V = f.V, P = sh.lanes;
  const int lane = threadIdx.x & 31, warp = __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0), nwarps = blockDim.x >> 5;
  {
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw + f.pool_bytes);
    if (!stage_blob(smem_raw, fblob + f.prec, f.pool_bytes, bar, err)) return;
  }
  const uint32_t smem_a = smem_u32(smem_raw), more_a = smem_a + f.pmore;
  const uint16_t* roots = reinterpret_cast<const uint16_t*>(smem_raw + f.roots);
  const uint8_t* first = smem_raw + f.joins;
  const uint32_t mine = smem_a + sh.off_state + (uint32_t)warp * sh.state_bytes;
  const uint32_t pool_a = mine + (uint32_t)lane * 16u, qpitch = (uint32_t)P * 16u;   // bytes of a row of four places
  const uint32_t rank_a = mine + sh.off_rank + (uint32_t)lane * 2u, rpitch = (uint32_t)P * 2u;
  const uint32_t cnt_a = mine + sh.off_cnt + (uint32_t)lane, cpitch = (uint32_t)P;
  auto place_at = [&](uint32_t t) { return pool_a + (t >> 2) * qpitch + (t & 3u) * 4u; };
  const uint32_t K2 = (uint32_t)K * 2u, joins = (uint32_t)f.num_joins, vlast = (uint32_t)(V - 1);

  for (int64_t tile = (int64_t)warp * gridDim.x + blockIdx.x; tile < sh.tiles; tile += (int64_t)nwarps * gridDim.x) {
    const int64_t c = tile * P + lane;
    if (lane >= P || c >= K) continue;   // (the lanes of a warp have nothing to do with each other)
#pragma unroll
    for (int q = 0; q < QUADS; ++q) sts128(pool_a + (uint32_t)q * qpitch, make_uint4(kNoKey, kNoKey, kNoKey, kNoKey));
    for (int i = 0; i < V; ++i) sts16(rank_a + (uint32_t)i * rpitch, 0xFFFFu);
    for (uint32_t j = 0; j < joins + 1u; ++j) sts8(cnt_a + j * cpitch, j < joins ? (uint32_t)first[j] : 0u);

    // the list: the operators' ranks; an operator twice, or an entry that is none, leaves another one out
    {
      const uint8_t* at = reinterpret_cast<const uint8_t*>(list + c);
      constexpr int kBatch = 64;   // (few warps: what is in flight decides; rows of 16 took 40 us at V = 1536)
      int r0 = 0;
      for (; r0 + kBatch <= V; r0 += kBatch) {
        uint32_t i[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) i[u] = __ldg(reinterpret_cast<const uint16_t*>(at + (uint64_t)(uint32_t)(r0 + u) * K2));
#pragma unroll
        for (int u = 0; u < kBatch; ++u)
          if (i[u] < (uint32_t)V) sts16(rank_a + i[u] * rpitch, (uint32_t)(r0 + u));
      }
#pragma unroll 8
      for (; r0 < V; ++r0) {
        const uint32_t i = __ldg(reinterpret_cast<const uint16_t*>(at + (uint64_t)(uint32_t)r0 * K2));
        if (i < (uint32_t)V) sts16(rank_a + i * rpitch, (uint32_t)r0);
      }
    }
    uint32_t most = 0;
#pragma unroll 16
    for (int i = 0; i < V; ++i) most = max(most, lds16(rank_a + (uint32_t)i * rpitch));
    const bool bad = most == 0xFFFFu;
    if (status) status[c] = bad ? (uint32_t)PE_STATUS_ORDER_INVALID : 0u;
    if (bad) continue;   // not a permutation: the order of this candidate stays unwritten

    uint32_t open = f.num_roots < 32 ? ~0u << f.num_roots : 0u;   // free places
    for (uint32_t t = 0; t < (uint32_t)f.num_roots; ++t) {
      const uint32_t i = roots[t];
      sts32(place_at(t), lds16(rank_a + i * rpitch) << 17 | t << 12 | i);
    }
    uint8_t* out = reinterpret_cast<uint8_t*>(order + c);
    int k = 0;
    uint32_t left = 0, succ = 0xFFFF0000u, more = more_a;   // of the operator placed last: successors to come, the next one, where the others are
    for (int it = 0; it < f.turns + 1 && k < V; ++it) {     // (one turn a successor, one for an operator without, one to begin with)
      const bool has = left != 0u;
      const uint32_t s = succ & 0xFFFFu, j = succ >> 16;
      const bool join = j != 0xFFFFu;
      const uint32_t r = lds16(rank_a + s * rpitch);
      const uint32_t m = lds8(cnt_a + (join ? j : joins) * cpitch);
      const uint32_t succ_more = lds32(more);
      uint4 p[QUADS];
#pragma unroll
      for (int q = 0; q < QUADS; ++q) p[q] = lds128(pool_a + (uint32_t)q * qpitch);
      sts8(cnt_a + (join && has ? j : joins + 1u) * cpitch, m - 1u);
      const bool freed = has && m == 0u;
      const uint32_t t = (uint32_t)__ffs((int)open) - 1u;
      const uint32_t fresh = r << 17 | t << 12 | s;
      sts32_if(place_at(t & 31u), fresh, freed);
      open = freed ? open & (open - 1u) : open;
      left -= has ? 1u : 0u;
      succ = succ_more;
      more += has ? 4u : 0u;
      uint32_t rest[QUADS];
#pragma unroll
      for (int q = 0; q < QUADS; ++q) rest[q] = min(min(p[q].x, p[q].y), min(p[q].z, p[q].w));
#pragma unroll
      for (int q = 1; q < QUADS; ++q) rest[0] = min(rest[0], rest[q]);
      const uint32_t key = min(rest[0], freed ? fresh : kNoKey);
      const bool pop = left == 0u;   // (some operator is available until the last one is placed)
      const uint32_t i = min(key & 0xFFFu, vlast), at = (key >> 12) & 31u;
      sts32_if(place_at(at), kNoKey, pop);
      const uint2 rec = lds64(smem_a + i * 8u);
      if (pop) *reinterpret_cast<uint16_t*>(out) = (uint16_t)i;
      out += pop ? K2 : 0u;
      k += pop ? 1 : 0;
      open |= pop ? 1u << at : 0u;
      succ = pop ? rec.x : succ;
      left = pop ? rec.y >> 24 : left;
      more = pop ? more_a + (rec.y & 0xFFFFFFu) * 4u : more;
    }
  }
}

struct DecodePlan {
  bool shared = false;      // per-operator state on chip
  bool lane = false;        // pe_decode_lane_kernel
  bool pool = false;        // pe_decode_pool_kernel, otherwise pe_decode_warp_kernel
  PoolShape shape = {};
  int64_t grid = 0;
  double us = 1e30;         // estimated time
  bool rec_smem = false;    // operator records in shared memory
  int threads = 0;
  uint32_t words = 0;       // shared words per warp
  size_t smem = 0;
  size_t workspace = 0;
};

static bool plan_decode_warp(const pe_graph* g, int64_t K, DecodePlan* p) {
  const size_t V = (size_t)g->V, n0 = (V + 31) / 32, rb = g->fview.rec_bytes;
  if (V > 65535) return false;
  // the block size that keeps most warps on an SM, and no more warps per block than spread the batch over the SMs
  size_t best = 0;
  for (size_t nw = 1; nw <= 8; nw *= 2) {
    if (nw > 1 && (int64_t)nw * g->sm_count > K) break;
    const bool with = V * rb <= kDecodeRecBytes;
    const size_t words = (V + 1 + n0 + 32 + 3) / 4 * 4;
    const size_t bytes = nw * words * 4 + (with ? V * rb : 0);
    if (bytes > g->smem_optin) break;
    size_t blocks = g->smem_per_sm / (bytes + 1024);
    if (blocks > 32) blocks = 32;
    const size_t warps = std::min<size_t>(blocks * nw, 64);
    if (warps <= best) continue;
    best = warps;
    p->rec_smem = with;
    p->threads = (int)(32 * nw);
    p->words = (uint32_t)words;
    p->smem = bytes;
  }
  p->shared = best > 0;
  // bound by issue, or by the chain of a placement (longer where the records are not on chip).  Measured (estimate / time, us):
  // V = 64 K = 64 16.9 / 16.4, V = 704 K = 256 111 / 119, V = 1536 K = 1024 233 / 240, K = 16384 1426 / 1524; records not on
  // chip: V = 2304 K = 256 479 / 479, V = 2816 K = 256 692 / 682, K = 8192 2865 / 2785.
  const double dV = (double)V, dK = (double)K, dE = (double)g->fview.E, per_sm = std::max(1.0, dK / (double)g->sm_count);
  if (best > 0)
    p->us = 7.5 + std::max(dV * dK * (55.0 + 1.4 * dE / dV) * 1e-6,
                           (p->rec_smem ? 0.147 * dV : 0.145 * dV + 0.06 * dE) * per_sm / std::min(per_sm, (double)best));
  return p->shared;
}

static bool plan_decode_lane(const pe_graph* g, int64_t K, DecodePlan* p) {
  const size_t V = (size_t)g->V, E = (size_t)g->fview.E;
  if (V > 256 || E > 65535 || !g->fview.short_lists) return false;
  const size_t bytes = V * 4 + (V + 31) / 32 * kLaneThreads * 4 + V * kLaneThreads * 3 + (E + 3) / 4 * 4;
  if (bytes > g->smem_optin) return false;
  // A lane takes ~0.1 us a placement and ~0.3 us a successor, less (~0.12 us) for those beyond two an operator, which come
  // without a placement of their own, however few candidates there are; the candidates that fit on chip go through in
  // rounds.  The warp kernel places ~18000 operators a microsecond, the fewer the more successors they have.  Measured (lane
  // / warp, us): V = 64, E = 56 K = 8192 28 / 39, K = 32768 31 / 126; V = 256, E = 483 K = 8192 181 / 135, K = 32768 188 /
  // 446; V = 64, E = 819 K = 16384 108 / 88, K = 65536 122 / 311; V = 256, E = 6200 K = 65536 1696 / 1463; V = 128, E = 4146
  // K = 131072 893 / 1667.
  const double dV = (double)V, dE = (double)E, paired = std::min(dE, 2.0 * dV);
  const int64_t resident = (int64_t)(g->smem_per_sm / (bytes + 1024)) * kLaneThreads * g->sm_count;
  const double rounds = resident > 0 ? (double)((K + resident - 1) / resident) : 1e30;
  const double by_lane = (0.1 * dV + 0.3 * paired + 0.12 * (dE - paired)) * rounds;
  const double by_warp = 6.0 + dV * (double)K * (55.0 + 1.4 * dE / dV) * 1e-6;
  if (by_lane > by_warp) return false;
  p->us = by_lane;
  p->shared = p->lane = true;
  p->threads = kLaneThreads;
  p->smem = bytes;
  return true;
}

// A turn is a chain of shared-memory round trips, longer with more places to read, and bound by issue from five warps on an SM
// on.  Measured (estimate / time, us): V = 64 K = 1024 15.2 / 14.3, K = 65536 28 / 27; V = 704 (MoE) K = 8192 143 / 137; V = 1536
// K = 8192 196 / 199, K = 16384 384 / 389; V = 2304 K = 4096 309 / 315; V = 2816 K = 4096 627 / 633, K = 16384 2484 / 2510.
static bool plan_decode_pool(const pe_graph* g, int64_t K, DecodePlan* p) {
  const PeFwdView& f = g->fview;
  if (!f.pool_bytes || K < 1 || K >= ((int64_t)1 << 30)) return false;
  const size_t V = (size_t)g->V, fixed = ((size_t)f.pool_bytes + 8 + 15) / 16 * 16;
  auto bytes = [&](size_t P) { return (P * (4 * (size_t)f.places + 2 * V + (size_t)f.num_joins + 2) + 15) / 16 * 16; };
  size_t bestW = 0, bestP = 0;
  double best = 0;
  for (size_t W = 1; W <= 16; ++W)
    for (size_t P = 32; P >= 4; P -= 4)
      if (fixed + W * bytes(P) <= g->smem_optin) {
        const double score = (double)(W * P) / (W <= 4 ? 1.0 : 1.0 + 0.14 * (double)(W - 4));   // (narrow tiles of many warps cost)
        if (score > best) { best = score; bestW = W; bestP = P; }
        break;
      }
  if (bestW == 0) return false;
  const int64_t sms = g->sm_count, tiles = (K + (int64_t)bestP - 1) / (int64_t)bestP;
  const int64_t rounds = (tiles + sms * (int64_t)bestW - 1) / (sms * (int64_t)bestW);
  const int64_t w = (tiles + sms * rounds - 1) / (sms * rounds);
  if (w < (int64_t)bestW) bestW = (size_t)w;
  const double turn = std::max(0.092 + 0.0011 * f.places, 0.021 * (double)bestW);
  p->us = 8.0 + (0.012 * (double)V + turn * (double)f.turns) * (double)rounds;
  p->shared = p->pool = true;
  p->rec_smem = false;
  p->threads = (int)(32 * bestW);
  p->grid = std::min(tiles, sms);
  PoolShape& sh = p->shape;
  sh.lanes = (int)bestP;
  sh.tiles = tiles;
  sh.off_state = (uint32_t)fixed;
  sh.state_bytes = (uint32_t)bytes(bestP);
  sh.off_rank = (uint32_t)(bestP * 4 * (size_t)f.places);
  sh.off_cnt = sh.off_rank + (uint32_t)((bestP * 2 * V + 3) / 4 * 4);
  p->smem = fixed + bestW * bytes(bestP);
  return true;
}

static bool decode_plan(const pe_graph* g, int64_t K, uint32_t flags, DecodePlan* p) {
  if (!g->fwd_ok) return false;
  const uint32_t want = flags & PE_VARIANT_MASK;
  const size_t V = (size_t)g->V, n0 = (V + 31) / 32, n1 = (n0 + 31) / 32;
  if (want == PE_VARIANT_AUTO || want == PE_VARIANT_SHARED) {
    DecodePlan pool;
    if (!plan_decode_lane(g, K, p)) plan_decode_warp(g, K, p);
    if (plan_decode_pool(g, K, &pool) && 1.08 * pool.us < p->us) *p = pool;   // (what the estimates are off by)
    if (p->shared) return true;
    if (want == PE_VARIANT_SHARED) return false;
  }
  if (want != PE_VARIANT_AUTO && want != PE_VARIANT_GLOBAL) return false;
  p->shared = false;
  p->threads = 128;
  p->smem = 0;
  p->workspace = (size_t)((K + 31) / 32) * (V + n0 + n1) * 32 * 4;
  p->workspace = (p->workspace + 255) / 256 * 256;
  return true;
}

}  // namespace pe

extern "C" size_t pe_decode_workspace_bytes(const pe_graph* g, int64_t K, uint32_t flags) {
  pe::DecodePlan p;
  if (!g || K < 0 || !pe::decode_plan(g, K, flags, &p)) return 0;
  return p.workspace;
}

extern "C" int pe_decode_variant(const pe_graph* g, int64_t K, uint32_t flags) {
  pe::DecodePlan p;
  if (!g || K < 0) return PE_ERR_INVALID_ARG;
  if (flags & ~(uint32_t)PE_VARIANT_MASK) return PE_ERR_INVALID_ARG;
  if (!pe::decode_plan(g, K, flags, &p)) return PE_ERR_UNSUPPORTED;
  return p.shared ? PE_VARIANT_SHARED : PE_VARIANT_GLOBAL;
}

extern "C" int pe_decode_priority(pe_graph* g, int64_t K, const void* list, int order_bytes, uint32_t flags, void* order,
                                  uint32_t* status, void* workspace, size_t workspace_bytes, void* cuda_stream) {
  if (!g || K < 0) return PE_ERR_INVALID_ARG;
  if (flags & ~(uint32_t)PE_VARIANT_MASK) return PE_ERR_INVALID_ARG;
  if (order_bytes != 2 && order_bytes != 4) return PE_ERR_INVALID_ARG;
  if (order_bytes != 2) return PE_ERR_UNSUPPORTED;
  pe::DecodePlan p;
  if (!pe::decode_plan(g, K, flags, &p)) return PE_ERR_UNSUPPORTED;
  if (K == 0) return PE_OK;
  if (!list || !order) return PE_ERR_INVALID_ARG;
  if (K > (int64_t)INT_MAX) return PE_ERR_INVALID_ARG;
  if (p.workspace > 0 && (!workspace || workspace_bytes < p.workspace)) return PE_ERR_WORKSPACE;
  int prev = -1;
  if (cudaGetDevice(&prev) != cudaSuccess) return PE_ERR_CUDA;
  if (prev != g->device && cudaSetDevice(g->device) != cudaSuccess) return PE_ERR_CUDA;
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  const uint16_t* list16 = static_cast<const uint16_t*>(list);
  uint16_t* order16 = static_cast<uint16_t*>(order);
  int ret = PE_OK;
  if (p.lane) {
    auto kern = pe::pe_decode_lane_kernel;
    if (!pe::set_smem(kern, p.smem)) ret = PE_ERR_CUDA;
    else kern<<<(unsigned)((K + p.threads - 1) / p.threads), p.threads, p.smem, stream>>>(g->fview, g->d_fwd, K, list16, order16, status);
  } else if (p.pool) {
    auto kern = g->fview.places <= 8 ? pe::pe_decode_pool_kernel<2> : (g->fview.places <= 16 ? pe::pe_decode_pool_kernel<4> : (g->fview.places <= 24 ? pe::pe_decode_pool_kernel<6> : pe::pe_decode_pool_kernel<8>));
    if (!pe::set_smem(kern, p.smem)) ret = PE_ERR_CUDA;
    else kern<<<(unsigned)p.grid, p.threads, p.smem, stream>>>(g->fview, g->d_fwd, K, list16, order16, status, p.shape, g->d_error);
  } else if (p.shared) {
    const int64_t nw = p.threads / 32;
    auto kern = p.rec_smem ? pe::pe_decode_warp_kernel<true> : pe::pe_decode_warp_kernel<false>;
    if (!pe::set_smem(kern, p.smem)) ret = PE_ERR_CUDA;
    else kern<<<(unsigned)((K + nw - 1) / nw), p.threads, p.smem, stream>>>(g->fview, g->d_fwd, K, list16, order16, status, p.words);
  } else {
    pe::pe_decode_kernel<<<(unsigned)((K + p.threads - 1) / p.threads), p.threads, 0, stream>>>(
        g->fview, g->d_fwd, K, list16, order16, status, static_cast<uint32_t*>(workspace));
  }
  if (ret == PE_OK) {
    pe::g_decode_launches.fetch_add(1, std::memory_order_relaxed);
    if (cudaGetLastError() != cudaSuccess) ret = PE_ERR_CUDA;
  }
  if (prev != g->device) cudaSetDevice(prev);
  return ret;
}
