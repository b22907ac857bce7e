// pe_select_best: arg-min of the makespan (Eq. 1) over the candidates that pass the status mask.
#include <atomic>
#include <climits>

#include "pe.h"
#include "pe_launch.h"
#include <cuda_runtime.h>

namespace pe {

// key = makespan << 32 | index: the 64-bit minimum is the smallest makespan, ties to the smallest index
constexpr unsigned long long kNoKey = ~0ull;

// The four result words double as the running state: [0] minimum key, [2] qualifying candidates,
// [3] blocks finished; the last block to finish turns [0] into {index, makespan} in [0], [1].
__global__ void pe_select_init_kernel(unsigned long long* r) {
  r[0] = kNoKey;
  r[1] = 0ull;
  r[2] = 0ull;
  r[3] = 0ull;
}

__global__ void __launch_bounds__(256) pe_select_kernel(int64_t K, const int32_t* __restrict__ makespan,
                                                        const uint32_t* __restrict__ status, uint32_t reject_mask,
                                                        unsigned long long* scratch) {
  unsigned long long best = kNoKey;
  unsigned long long count = 0;
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < K; c += (int64_t)gridDim.x * blockDim.x) {
    if ((status[c] & reject_mask) == 0) {
      ++count;
      const unsigned long long key = ((unsigned long long)(unsigned)makespan[c] << 32) | (unsigned long long)c;
      best = key < best ? key : best;
    }
  }
  for (int off = 16; off > 0; off >>= 1) {
    const unsigned long long o = __shfl_xor_sync(0xFFFFFFFFu, best, off);
    best = o < best ? o : best;
    count += __shfl_xor_sync(0xFFFFFFFFu, count, off);
  }
  __shared__ unsigned long long s_best[8], s_count[8];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) { s_best[warp] = best; s_count[warp] = count; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
      best = s_best[w] < best ? s_best[w] : best;
      count += s_count[w];
    }
    if (best != kNoKey) atomicMin(&scratch[0], best);
    if (count) atomicAdd(&scratch[2], count);
    __threadfence();
    const unsigned long long done = atomicAdd(&scratch[3], 1ull) + 1ull;
    if (done == gridDim.x) {  // the last block publishes the result
      __threadfence();
      const unsigned long long m = atomicMin(&scratch[0], kNoKey);  // atomic read
      int64_t* result = reinterpret_cast<int64_t*>(scratch);
      result[0] = m == kNoKey ? -1 : (int64_t)(m & 0xFFFFFFFFull);
      result[1] = m == kNoKey ? (int64_t)INT32_MAX : (int64_t)(m >> 32);
    }
  }
}

// Batches up to these sizes are handled by one block: no state to set up, one launch.  (us, one block / many: best of 24576
// 6.3 / 7.1, of 28000 8.3 / 6.9; the k best of 32768 14.4 / 51)
constexpr int64_t kOneBlockBest = 24576, kOneBlock = 32768;

__global__ void __launch_bounds__(1024) pe_select_one_kernel(int K, const int32_t* __restrict__ makespan,
                                                             const uint32_t* __restrict__ status, uint32_t reject_mask,
                                                             int64_t* result) {
  unsigned long long best = kNoKey;
  unsigned int count = 0;
#pragma unroll 8
  for (int c = threadIdx.x; c < K; c += 1024) {
    const uint32_t s = status[c];
    const int32_t m = makespan[c];
    if ((s & reject_mask) == 0) {
      ++count;
      const unsigned long long key = ((unsigned long long)(unsigned)m << 32) | (unsigned long long)c;
      best = key < best ? key : best;
    }
  }
  __shared__ unsigned long long s_best[32];
  __shared__ unsigned int s_count[32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int round = 0; round < 2; ++round) {
    for (int off = 16; off > 0; off >>= 1) {
      const unsigned long long o = __shfl_xor_sync(0xFFFFFFFFu, best, off);
      best = o < best ? o : best;
    }
    count = __reduce_add_sync(0xFFFFFFFFu, count);
    if (round == 1 || warp >= 32) break;
    if (lane == 0) { s_best[warp] = best; s_count[warp] = count; }
    __syncthreads();
    best = s_best[lane];
    count = s_count[lane];
  }
  if (threadIdx.x == 0) {
    result[0] = best == kNoKey ? -1 : (int64_t)(best & 0xFFFFFFFFull);
    result[1] = best == kNoKey ? (int64_t)INT32_MAX : (int64_t)(best >> 32);
    result[2] = (int64_t)count;
    result[3] = 0;
  }
}

}  // namespace pe

extern "C" int pe_select_best(int64_t K, const int32_t* makespan, const uint32_t* status, uint32_t reject_mask,
                              int64_t* result, void* cuda_stream) {
  if (K < 0 || !result || (K > 0 && (!makespan || !status))) return PE_ERR_INVALID_ARG;
  if (K > 0xFFFFFFFFll) return PE_ERR_INVALID_ARG;  // the index shares a 64-bit key with the makespan
  // run on the device that owns `result` (the other arrays must live there too)
  cudaPointerAttributes attr;
  if (cudaPointerGetAttributes(&attr, result) != cudaSuccess ||
      (attr.type != cudaMemoryTypeDevice && attr.type != cudaMemoryTypeManaged)) {
    cudaGetLastError();
    return PE_ERR_INVALID_ARG;
  }
  int prev = -1;
  if (cudaGetDevice(&prev) != cudaSuccess) return PE_ERR_CUDA;
  if (prev != attr.device && cudaSetDevice(attr.device) != cudaSuccess) return PE_ERR_CUDA;
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  unsigned long long* scratch = reinterpret_cast<unsigned long long*>(result);
  if (K <= pe::kOneBlockBest) {
    pe::pe_select_one_kernel<<<1, 1024, 0, stream>>>((int)K, makespan, status, reject_mask, result);
  } else {
    pe::pe_select_init_kernel<<<1, 1, 0, stream>>>(scratch);
    const int64_t want = (K + 255) / 256;
    const int blocks = (int)(want < 1184 ? want : 1184);  // 148 SMs x 8 resident blocks: a grid-stride loop covers the rest
    pe::pe_select_kernel<<<blocks, 256, 0, stream>>>(K, makespan, status, reject_mask, scratch);
  }
  const int ret = cudaGetLastError() == cudaSuccess ? PE_OK : PE_ERR_CUDA;
  if (prev != attr.device) cudaSetDevice(prev);
  return ret;
}

// ============================================================================================
// pe_select_topk: the k best qualifying candidates (smallest makespan, ties to the smallest index).
//
// Radix select on the makespan (three passes over 11 + 11 + 10 bits) finds the value T of the k-th best
// and how many candidates are strictly better; an ordered compaction (per-block counts, a scan over
// the blocks, a write pass) then lists, by increasing index, every candidate better than T and the
// first (k - better) candidates equal to T.  State lives in the caller's workspace:
//   words [0..7]   : prefix (bits of T fixed so far), remaining rank, qualifying count, result count
//   words [8..]    : histogram (2048 bins), then per-block (better, equal) counts and their scans
// ============================================================================================
namespace pe {

constexpr int kTopkBins = 2048;
constexpr int kTopkBlock = 256;
constexpr int kTopkPerBlock = 4096;   // candidates per block of the compaction passes

struct TopkState {
  unsigned int prefix;      // high bits of T found so far
  unsigned int remaining;   // rank still to resolve inside the current prefix (1-based)
  unsigned int qualifying;  // candidates that pass the mask
  unsigned int take_equal;  // how many candidates equal to T belong to the result
  unsigned int threshold;   // T
  unsigned int none;        // 1 when fewer than k qualify: everything qualifying is taken
  unsigned int pad[2];
};

__global__ void pe_topk_init_kernel(TopkState* s, unsigned int* hist, unsigned int k) {
  for (int b = threadIdx.x; b < kTopkBins; b += blockDim.x) hist[b] = 0;
  if (threadIdx.x == 0) {
    s->prefix = 0; s->remaining = k; s->qualifying = 0; s->take_equal = 0; s->threshold = 0; s->none = 0;
  }
}

// histogram of the `bits` bits at `shift` over the qualifying candidates whose higher bits equal the prefix
__global__ void __launch_bounds__(kTopkBlock) pe_topk_hist_kernel(int64_t K, const int32_t* __restrict__ makespan,
                                                                  const uint32_t* __restrict__ status,
                                                                  uint32_t reject_mask, const TopkState* s,
                                                                  unsigned int* hist, int shift, int bits, int first) {
  __shared__ unsigned int sh[kTopkBins];
  for (int b = threadIdx.x; b < kTopkBins; b += blockDim.x) sh[b] = 0;
  __syncthreads();
  const unsigned int prefix = s->prefix;
  const unsigned int mask = (1u << bits) - 1u;
  unsigned int qual = 0;
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < K; c += (int64_t)gridDim.x * blockDim.x) {
    if ((status[c] & reject_mask) != 0) continue;
    ++qual;
    const unsigned int v = (unsigned int)makespan[c];
    const int hi = shift + bits;
    if (hi < 32 && (v >> hi) != (prefix >> hi)) continue;
    atomicAdd(&sh[(v >> shift) & mask], 1u);
  }
  __syncthreads();
  for (int b = threadIdx.x; b < kTopkBins; b += blockDim.x)
    if (sh[b]) atomicAdd(&hist[b], sh[b]);
  if (first) {
    for (int off = 16; off > 0; off >>= 1) qual += __shfl_xor_sync(0xFFFFFFFFu, qual, off);
    if ((threadIdx.x & 31) == 0 && qual) atomicAdd(const_cast<unsigned int*>(&s->qualifying), qual);
  }
}

// one block: find the bin that holds the remaining-th smallest, fix its bits in the prefix, clear the histogram
__global__ void __launch_bounds__(kTopkBlock) pe_topk_pick_kernel(TopkState* s, unsigned int* hist, int shift, int bits,
                                                                  int first, int last) {
  __shared__ unsigned int part[kTopkBlock];
  __shared__ unsigned int chosen_bin, chosen_below;
  const int nb = 1 << bits;
  const int per = (nb + kTopkBlock - 1) / kTopkBlock;   // consecutive bins per thread
  if (first && threadIdx.x == 0 && s->qualifying < s->remaining) s->none = 1;
  __syncthreads();
  const bool none = s->none != 0;
  unsigned int mine = 0;
  for (int q = 0; q < per; ++q) {
    const int b = threadIdx.x * per + q;
    if (b < nb) mine += hist[b];
  }
  part[threadIdx.x] = mine;
  __syncthreads();
  if (threadIdx.x == 0 && !none) {
    unsigned int below = 0, rem = s->remaining;
    int t = 0;
    while (t < kTopkBlock - 1 && below + part[t] < rem) { below += part[t]; ++t; }
    int b = t * per;
    while (b < nb - 1 && below + hist[b] < rem) { below += hist[b]; ++b; }
    chosen_bin = (unsigned int)b;
    chosen_below = below;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (none) {
      s->threshold = 0xFFFFFFFFu;   // everything that qualifies is better than T
      s->take_equal = 0;
    } else {
      s->prefix |= chosen_bin << shift;
      s->remaining -= chosen_below;
      if (last) { s->threshold = s->prefix; s->take_equal = s->remaining; }
    }
  }
  __syncthreads();
  for (int b = threadIdx.x; b < kTopkBins; b += blockDim.x) hist[b] = 0;
}

// per block of kTopkPerBlock candidates: how many are better than T, how many equal
__global__ void __launch_bounds__(kTopkBlock) pe_topk_count_kernel(int64_t K, const int32_t* __restrict__ makespan,
                                                                   const uint32_t* __restrict__ status,
                                                                   uint32_t reject_mask, const TopkState* s,
                                                                   unsigned int* blk) {
  const unsigned int T = s->threshold;
  unsigned int better = 0, equal = 0;
  const int64_t base = (int64_t)blockIdx.x * kTopkPerBlock;
  for (int q = threadIdx.x; q < kTopkPerBlock; q += kTopkBlock) {
    const int64_t c = base + q;
    if (c < K && (status[c] & reject_mask) == 0) {
      const unsigned int v = (unsigned int)makespan[c];
      better += v < T;
      equal += v == T;
    }
  }
  for (int off = 16; off > 0; off >>= 1) {
    better += __shfl_xor_sync(0xFFFFFFFFu, better, off);
    equal += __shfl_xor_sync(0xFFFFFFFFu, equal, off);
  }
  __shared__ unsigned int sb[kTopkBlock / 32], se[kTopkBlock / 32];
  if ((threadIdx.x & 31) == 0) { sb[threadIdx.x >> 5] = better; se[threadIdx.x >> 5] = equal; }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned int b = 0, e = 0;
    for (int w = 0; w < kTopkBlock / 32; ++w) { b += sb[w]; e += se[w]; }
    blk[2 * blockIdx.x] = b;
    blk[2 * blockIdx.x + 1] = e;
  }
}

// one block: exclusive scan of the per-block counts, in place
__global__ void __launch_bounds__(kTopkBlock) pe_topk_scan_kernel(unsigned int* blk, int nblocks) {
  __shared__ unsigned int sb[kTopkBlock], se[kTopkBlock];
  __shared__ unsigned int carry_b, carry_e;
  if (threadIdx.x == 0) { carry_b = 0; carry_e = 0; }
  __syncthreads();
  for (int base = 0; base < nblocks; base += kTopkBlock) {
    const int i = base + threadIdx.x;
    const unsigned int b = i < nblocks ? blk[2 * i] : 0u, e = i < nblocks ? blk[2 * i + 1] : 0u;
    sb[threadIdx.x] = b; se[threadIdx.x] = e;
    __syncthreads();
    for (int off = 1; off < kTopkBlock; off <<= 1) {   // inclusive scan of the chunk
      const unsigned int pb = threadIdx.x >= off ? sb[threadIdx.x - off] : 0u;
      const unsigned int pe_ = threadIdx.x >= off ? se[threadIdx.x - off] : 0u;
      __syncthreads();
      sb[threadIdx.x] += pb; se[threadIdx.x] += pe_;
      __syncthreads();
    }
    if (i < nblocks) { blk[2 * i] = carry_b + sb[threadIdx.x] - b; blk[2 * i + 1] = carry_e + se[threadIdx.x] - e; }
    __syncthreads();
    if (threadIdx.x == 0) { carry_b += sb[kTopkBlock - 1]; carry_e += se[kTopkBlock - 1]; }
    __syncthreads();
  }
}

// A candidate is taken if it is better than T, or equal to T with fewer than take_equal equal ones before it.
// Its place in the output is the number of taken candidates before it, which is
// better_before + min(equal_before, take_equal): the list comes out ordered by candidate index.
__global__ void __launch_bounds__(kTopkBlock) pe_topk_write_kernel(int64_t K, const int32_t* __restrict__ makespan,
                                                                   const uint32_t* __restrict__ status,
                                                                   uint32_t reject_mask, const TopkState* s,
                                                                   const unsigned int* blk, int32_t k,
                                                                   int32_t* out_index, int32_t* out_count) {
  constexpr int kPer = kTopkPerBlock / kTopkBlock;   // consecutive candidates per thread
  const unsigned int T = s->threshold, take_equal = s->take_equal;
  const int64_t first = (int64_t)blockIdx.x * kTopkPerBlock + (int64_t)threadIdx.x * kPer;
  unsigned int flag_b = 0, flag_e = 0, nb = 0, ne = 0;
  for (int q = 0; q < kPer; ++q) {
    const int64_t c = first + q;
    if (c < K && (status[c] & reject_mask) == 0) {
      const unsigned int v = (unsigned int)makespan[c];
      if (v < T) { flag_b |= 1u << q; ++nb; }
      if (v == T) { flag_e |= 1u << q; ++ne; }
    }
  }
  // exclusive scan of (nb, ne) over the block's threads
  unsigned int pb = nb, pe_ = ne;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int off = 1; off < 32; off <<= 1) {
    const unsigned int ub = __shfl_up_sync(0xFFFFFFFFu, pb, off), ue = __shfl_up_sync(0xFFFFFFFFu, pe_, off);
    if (lane >= off) { pb += ub; pe_ += ue; }
  }
  __shared__ unsigned int wb[kTopkBlock / 32], we[kTopkBlock / 32];
  if (lane == 31) { wb[warp] = pb; we[warp] = pe_; }
  __syncthreads();
  unsigned int before_b = blk[2 * blockIdx.x] + pb - nb, before_e = blk[2 * blockIdx.x + 1] + pe_ - ne;
  for (int w = 0; w < warp; ++w) { before_b += wb[w]; before_e += we[w]; }
  for (int q = 0; q < kPer; ++q) {
    const bool isb = (flag_b >> q) & 1u, ise = (flag_e >> q) & 1u;
    if (isb || (ise && before_e < take_equal)) {
      const unsigned int at = before_b + (before_e < take_equal ? before_e : take_equal);
      if (at < (unsigned int)k) out_index[at] = (int32_t)(first + q);
    }
    before_b += isb;
    before_e += ise;
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == kTopkBlock - 1) {   // the totals end here
    const unsigned int total = before_b + (before_e < take_equal ? before_e : take_equal);
    *out_count = (int32_t)(total < (unsigned int)k ? total : (unsigned int)k);
  }
}

__global__ void pe_topk_fill_kernel(int32_t* out_index, int64_t from, int64_t k) {
  for (int64_t i = from + blockIdx.x * blockDim.x + threadIdx.x; i < k; i += gridDim.x * blockDim.x) out_index[i] = -1;
}
static void fill_rest(int32_t* out_index, int64_t from, int64_t k, cudaStream_t stream) {   // entries from .. k - 1
  if (k <= from) return;
  const int64_t want = (k - from + 255) / 256;
  pe_topk_fill_kernel<<<(unsigned)(want < 256 ? want : 256), 256, 0, stream>>>(out_index, from, k);
}

// The whole selection in one block, for batches whose keys fit in shared memory.  Bound by the latency of a few block
// barriers (a launch of its own per step, eleven in all, cost ~2 us each).  The histogram covers the range the values
// have, not 32 bits: most batches need one or two rounds, and neighbouring values do not meet in one bin.  Entries that
// cannot be filled are set to -1 up to `fill`; one block writes ~60 GB/s, so lists beyond kOneFill leave the rest to a
// launch with more blocks (K = 4096: k = 262144 22.6 -> 11.4 us, k = 4194304 272 -> 14.4 us; k = 40000 would take 10.4
// instead of 8.3 us that way).
constexpr int32_t kOneFill = 65536;
__global__ void __launch_bounds__(1024) pe_topk_one_kernel(int K, const int32_t* __restrict__ makespan,
                                                           const uint32_t* __restrict__ status, uint32_t reject_mask, int32_t k,
                                                           int32_t fill, int32_t* __restrict__ out_index,
                                                           int32_t* __restrict__ out_count) {
  extern __shared__ unsigned int keys[];   // makespan, or kNone where the candidate does not qualify
  constexpr unsigned int kNone = 0xFFFFFFFFu, FULL = 0xFFFFFFFFu;
  __shared__ unsigned int hist[kTopkBins];
  __shared__ unsigned int wa[32], wb[32], wc[32];
  __shared__ unsigned int sh_bin, sh_below;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  unsigned int lo = kNone, hi = 0, n = 0;
#pragma unroll 8
  for (int c = t; c < K; c += 1024) {
    const unsigned int m = (unsigned int)makespan[c];
    const unsigned int v = (status[c] & reject_mask) == 0 ? m : kNone;
    keys[c] = v;
    if (v != kNone) { lo = min(lo, v); hi = max(hi, v); ++n; }
  }
  lo = __reduce_min_sync(FULL, lo); hi = __reduce_max_sync(FULL, hi); n = __reduce_add_sync(FULL, n);
  if (lane == 0) { wa[warp] = lo; wb[warp] = hi; wc[warp] = n; }
  __syncthreads();
  lo = __reduce_min_sync(FULL, wa[lane]); hi = __reduce_max_sync(FULL, wb[lane]); n = __reduce_add_sync(FULL, wc[lane]);
  // T: the k-th smallest key; everything qualifying is better than it when at most k qualify
  unsigned int T = kNone, take_equal = 0;
  if (k > 0 && n > (unsigned int)k) {
    unsigned int base = lo, rem = (unsigned int)k;
    int bits = 32 - __clz((int)(hi - lo));
    while (true) {   // (each round fixes up to 11 bits: at most three)
      const int shift = bits > 11 ? bits - 11 : 0;
      __syncthreads();
      hist[t] = 0; hist[t + 1024] = 0;
      __syncthreads();
      const unsigned int range = bits >= 32 ? kNone : (1u << bits) - 1u;
      for (int c = t; c < K; c += 1024) {
        const unsigned int d = keys[c] - base;
        if (keys[c] != kNone && keys[c] >= base && d <= range) atomicAdd(&hist[d >> shift], 1u);
      }
      __syncthreads();
      const unsigned int h0 = hist[2 * t], h1 = hist[2 * t + 1];
      unsigned int incl = h0 + h1;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const unsigned int o = __shfl_up_sync(FULL, incl, off);
        incl += lane >= off ? o : 0u;
      }
      if (lane == 31) wa[warp] = incl;
      __syncthreads();
      incl += __reduce_add_sync(FULL, lane < warp ? wa[lane] : 0u);
      const unsigned int excl = incl - h0 - h1;
      if (excl < rem && incl >= rem) {   // exactly one thread: the bin that holds the rem-th smallest
        const bool first = excl + h0 >= rem;
        sh_bin = 2u * (unsigned int)t + (first ? 0u : 1u);
        sh_below = first ? excl : excl + h0;
      }
      __syncthreads();
      base += sh_bin << shift;
      rem -= sh_below;
      if (shift == 0) break;
      bits = shift;
    }
    T = base;
    take_equal = rem;
  }
  // ordered compaction: thread t owns consecutive candidates
  __syncthreads();
  const int per = ((K + 1023) / 1024) | 1;   // (odd: a warp's threads read different banks)
  const int c0 = min(t * per, K), c1 = min(c0 + per, K);
  unsigned int nb = 0, ne = 0;
  for (int c = c0; c < c1; ++c) { nb += keys[c] < T; ne += keys[c] == T && T != kNone; }
  unsigned int ib = nb, ie = ne;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const unsigned int ob = __shfl_up_sync(FULL, ib, off), oe = __shfl_up_sync(FULL, ie, off);
    ib += lane >= off ? ob : 0u;
    ie += lane >= off ? oe : 0u;
  }
  if (lane == 31) { wb[warp] = ib; wc[warp] = ie; }
  __syncthreads();
  const unsigned int xb = lane < 32 ? wb[lane] : 0u, xe = wc[lane];
  const unsigned int all = min((unsigned int)k, __reduce_add_sync(FULL, xb) + min(__reduce_add_sync(FULL, xe), take_equal));
  unsigned int before_b = ib - nb + __reduce_add_sync(FULL, lane < warp ? xb : 0u);
  unsigned int before_e = ie - ne + __reduce_add_sync(FULL, lane < warp ? xe : 0u);
  if (nb + ne)
    for (int c = c0; c < c1; ++c) {
      const bool better = keys[c] < T, equal = keys[c] == T && T != kNone;
      if (better || (equal && before_e < take_equal)) {
        const unsigned int at = before_b + min(before_e, take_equal);
        if (at < (unsigned int)k) out_index[at] = c;
      }
      before_b += better;
      before_e += equal;
    }
  for (int i = (int)all + t; i < fill; i += 1024) out_index[i] = -1;
  if (t == 0) *out_count = (int32_t)all;
}

static size_t topk_blocks(int64_t K) { return (size_t)((K + kTopkPerBlock - 1) / kTopkPerBlock); }

}  // namespace pe

extern "C" size_t pe_select_topk_workspace_bytes(int64_t K) {
  if (K < 0) return 0;
  return sizeof(pe::TopkState) + sizeof(unsigned int) * (pe::kTopkBins + 2 * (pe::topk_blocks(K) + 1));
}

extern "C" int pe_select_topk(int64_t K, const int32_t* makespan, const uint32_t* status, uint32_t reject_mask,
                              int32_t k, int32_t* out_index, int32_t* out_count, void* workspace,
                              size_t workspace_bytes, void* cuda_stream) {
  if (K < 0 || k < 0 || !out_count || (k > 0 && !out_index) || (K > 0 && (!makespan || !status))) return PE_ERR_INVALID_ARG;
  if (K > 0x7FFFFFFFll) return PE_ERR_INVALID_ARG;   // indices are int32
  if (!workspace || workspace_bytes < pe_select_topk_workspace_bytes(K) || ((uintptr_t)workspace & 15u))
    return PE_ERR_WORKSPACE;
  cudaPointerAttributes attr;
  if (cudaPointerGetAttributes(&attr, out_count) != cudaSuccess ||
      (attr.type != cudaMemoryTypeDevice && attr.type != cudaMemoryTypeManaged)) {
    cudaGetLastError();
    return PE_ERR_INVALID_ARG;
  }
  int prev = -1;
  if (cudaGetDevice(&prev) != cudaSuccess) return PE_ERR_CUDA;
  if (prev != attr.device && cudaSetDevice(attr.device) != cudaSuccess) return PE_ERR_CUDA;
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  pe::TopkState* st = static_cast<pe::TopkState*>(workspace);
  unsigned int* hist = reinterpret_cast<unsigned int*>(st + 1);
  unsigned int* blk = hist + pe::kTopkBins;
  const int nblocks = (int)pe::topk_blocks(K);
  int grid = (int)((K + pe::kTopkBlock - 1) / pe::kTopkBlock);
  if (grid > 1184) grid = 1184;
  if (grid < 1) grid = 1;
  if (K <= pe::kOneBlock) {
    int ret = PE_OK;
    const size_t bytes = sizeof(unsigned int) * (size_t)(K > 0 ? K : 1);
    if (!pe::set_smem(pe::pe_topk_one_kernel, bytes)) ret = PE_ERR_CUDA;
    else {
      const int32_t fill = k < pe::kOneFill ? k : pe::kOneFill;
      pe::fill_rest(out_index, fill, k, stream);
      pe::pe_topk_one_kernel<<<1, 1024, bytes, stream>>>((int)K, makespan, status, reject_mask, k, fill, out_index, out_count);
    }
    if (cudaGetLastError() != cudaSuccess) ret = PE_ERR_CUDA;
    if (prev != attr.device) cudaSetDevice(prev);
    return ret;
  }
  pe::fill_rest(out_index, 0, k, stream);
  pe::pe_topk_init_kernel<<<1, 256, 0, stream>>>(st, hist, (unsigned int)k);
  const int shifts[3] = {21, 10, 0}, bits[3] = {11, 11, 10};
  for (int p = 0; p < 3; ++p) {
    pe::pe_topk_hist_kernel<<<grid, pe::kTopkBlock, 0, stream>>>(K, makespan, status, reject_mask, st, hist, shifts[p],
                                                                 bits[p], p == 0);
    pe::pe_topk_pick_kernel<<<1, pe::kTopkBlock, 0, stream>>>(st, hist, shifts[p], bits[p], p == 0, p == 2);
  }
  {
    pe::pe_topk_count_kernel<<<nblocks, pe::kTopkBlock, 0, stream>>>(K, makespan, status, reject_mask, st, blk);
    pe::pe_topk_scan_kernel<<<1, pe::kTopkBlock, 0, stream>>>(blk, nblocks);
    pe::pe_topk_write_kernel<<<nblocks, pe::kTopkBlock, 0, stream>>>(K, makespan, status, reject_mask, st, blk, k,
                                                                      out_index, out_count);
  }
  const int ret = cudaGetLastError() == cudaSuccess ? PE_OK : PE_ERR_CUDA;
  if (prev != attr.device) cudaSetDevice(prev);
  return ret;
}
