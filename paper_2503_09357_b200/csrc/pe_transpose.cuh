// Tiled transposition between the candidate-interleaved arrays of the interface ([rows][K]) and
// candidate-major staging copies ([K][rows padded]).  A block of pe_eval_team_kernel works on one
// candidate; with the interleaved layout every one of its loads and stores would touch its own
// 32-byte sector (2 or 4 useful bytes each), with the staging copy it moves whole lines. The
// transposition itself reads whole 32-byte sectors (or more) and writes 128 contiguous bytes per warp instruction.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace pe {

// in:  [R][in_ld] elements of S bytes, columns 0..C-1 used; out: [C][out_ld], columns 0..R-1 written
// (and zeros up to the next multiple of 4 / S).  out_ld * S must be a multiple of 4 and `out` 4-byte aligned; `in` and
// its rows may start anywhere when !ALIGNED (odd batches: a word is put together from two aligned ones).
// One block of 128 threads moves a tile of 32 G rows by 32 columns (G = 4 / S elements per 32-bit word) through 4 KB of
// shared memory; word (r, cw) of the tile is kept at word (cw + r / G) mod (32 / G) of its row, which keeps the
// G-rows-per-lane reads to few lanes a bank.  grid = (ceil(C / 32), ceil(R / (32 G))).
// Bound by DRAM.  The tile is this small so that a few blocks fit next to the evaluation's blocks, which leave ~25 KB
// of an SM's shared memory and most of its threads free: the copies of one chunk then run while another is evaluated.
template <int S, bool ALIGNED>
__global__ void __launch_bounds__(128) pe_transpose_kernel(const uint8_t* __restrict__ in, uint8_t* __restrict__ out,
                                                           int64_t R, int64_t C, int64_t in_ld, int64_t out_ld) {
  constexpr int G = 4 / S;
  constexpr int TR = 32 * G;   // tile rows (elements)
  constexpr int TW = 32 / G;   // words of a tile row
  __shared__ uint32_t tile[TR][TW];
  const int64_t r0 = (int64_t)blockIdx.y * TR, c0 = (int64_t)blockIdx.x * 32;
  uint32_t* out_w = reinterpret_cast<uint32_t*>(out);
  const int64_t out_ldw = out_ld / G, rw0 = r0 / G;          // in words
  const int64_t Rw = (R + G - 1) / G;                        // words per output row
  const int64_t width = (C - c0) * S;                        // bytes of a row from the tile's first column on
  // load: consecutive threads take consecutive words of a row, then the next row
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int idx = q * 128 + threadIdx.x;
    const int r = idx / TW, cw = idx % TW;
    uint32_t w = 0;
    if (r0 + r < R && 4 * cw < width) {
      const uint8_t* at = in + ((r0 + r) * in_ld + c0) * S + 4 * cw;
      if (ALIGNED) {
        w = __ldg(reinterpret_cast<const uint32_t*>(at));
      } else {
        const uint32_t a = (uint32_t)(uintptr_t)at & 3u;
        const uint32_t* base = reinterpret_cast<const uint32_t*>(at - a);
        const uint32_t lo = __ldg(base), hi = (a != 0 && 4 * cw + 4 - (int)a < width) ? __ldg(base + 1) : 0u;
        w = __funnelshift_r(lo, hi, 8u * a);
      }
    }
    tile[r][(cw + r / G) % TW] = w;
  }
  __syncthreads();
  // store: word column cw of the tile holds G input columns; lane t owns input rows G t .. G t + G - 1
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int cw = warp; cw < TW; cw += 4) {
    uint32_t v[G];
#pragma unroll
    for (int q = 0; q < G; ++q) v[q] = tile[G * lane + q][(cw + lane) % TW];
    uint32_t o[G];
    if constexpr (G == 1) {
      o[0] = v[0];
    } else if constexpr (G == 2) {   // 2 x 2 halfwords
      o[0] = __byte_perm(v[0], v[1], 0x5410);
      o[1] = __byte_perm(v[0], v[1], 0x7632);
    } else {                         // 4 x 4 bytes
      const uint32_t t0 = __byte_perm(v[0], v[1], 0x5140), t1 = __byte_perm(v[2], v[3], 0x5140);
      const uint32_t t2 = __byte_perm(v[0], v[1], 0x7362), t3 = __byte_perm(v[2], v[3], 0x7362);
      o[0] = __byte_perm(t0, t1, 0x5410);
      o[1] = __byte_perm(t0, t1, 0x7632);
      o[2] = __byte_perm(t2, t3, 0x5410);
      o[3] = __byte_perm(t2, t3, 0x7632);
    }
#pragma unroll
    for (int q = 0; q < G; ++q) {
      const int64_t cc = c0 + (int64_t)G * cw + q;   // input column = output row
      if (cc < C && rw0 + lane < Rw) out_w[cc * out_ldw + rw0 + lane] = o[q];
    }
  }
}

}  // namespace pe
