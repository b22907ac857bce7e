// Internal: launch plan and the launchers of the compact-graph kernels (each family of
// kernel instantiations lives in its own translation unit so that they compile in parallel).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "pe_graph.h"
#include "pe_slot_shape.h"
#include "pe_tile_shape.h"

namespace pe {

struct Plan {
  int variant = 0;        // PE_VARIANT_* value
  int threads = 0;        // block size
  size_t smem = 0;        // dynamic shared memory per block
  bool graph_smem = false;  // graph blob staged into shared memory
  size_t workspace = 0;   // bytes of caller workspace
  size_t ws_x_off = 0;    // offset of the machine-state array inside the workspace (generic GLOBAL, by-pos)
  size_t ws_c_off = 0;    // generic GLOBAL with PE_COMM_EXCLUSIVE: offset of the per-channel array inside the workspace
  int warp_words = 0;     // WARP: 32-bit words of shared memory per candidate
  bool compact = false;   // SHARED / GLOBAL / WARP: the compact-graph kernels
  bool exclusive = false; // SHARED (compact): PE_COMM_EXCLUSIVE, one more word per machine pair and candidate
  bool slab = false;      // WARP (compact): order entries and times go through shared tiles, a slab at a time
  // SHARED over the tile encoding (pe_eval_tile_kernel)
  bool tiled = false;
  int tile_mode = 0;
  int tile_resident = 0;    // candidates an SM holds at once
  int64_t tile_rounds = 0;  // tiles that a warp evaluates one after the other
  int64_t grid = 0;
  TileShape tile = {};
  // SHARED over the slot encoding (pe_eval_slot_kernel; tile_mode, tile_resident, tile_rounds as above): candidates of a
  // chunk, row pitch and offsets of the workspace arrays, candidates per block of the kernels around it
  bool slot = false;
  int64_t slot_chunk = 0, slot_pitch = 0;
  size_t slot_off_status = 0, slot_off_wsum = 0, slot_off_words = 0;
  int slot_gather = 0, slot_times = 0;
  SlotShape slot_shape = {};
  // TEAM: inputs and times go through candidate-major staging copies in the workspace, a chunk of candidates at a time
  bool staged = false;
  int64_t team_chunk = 0;   // candidates per chunk
  int64_t team_vp = 0;      // row length of the staging copies: V rounded up to a multiple of 64
  size_t team_off_order = 0, team_off_assign = 0, team_off_start = 0, team_off_finish = 0;   // offsets in a half
  size_t team_half = 0;     // bytes of one half of the workspace (two chunks are in flight)
};

// Raise a kernel's dynamic shared-memory limit to at least `bytes` on the current device.  The attribute
// belongs to the function, not to a launch, and several host threads may launch the same kernel with
// different sizes: the limit is therefore only ever raised, under a lock, so a launch that was prepared
// with a smaller size can never find the limit lowered underneath it.
bool raise_smem_limit(const void* func, size_t bytes);

template <typename Kern>
static bool set_smem(Kern kern, size_t bytes) {
  return raise_smem_limit(reinterpret_cast<const void*>(kern), bytes);
}

// pe_eval_tile_kernel (plan variant SHARED over the tile encoding).
bool plan_tile(const pe_graph* g, int64_t K, bool by_pos, bool exclusive, Plan* p);
int launch_tile(const pe_graph* g, const Plan& p, bool by_pos, int64_t K, const uint8_t* assign, const uint16_t* order,
                uint32_t flags, const pe_outputs& out, cudaStream_t stream);

// pe_eval_slot_kernel (plan variant SHARED over the slot encoding) with the kernels around it; needs plan.workspace.
// Adds the number of kernels it launched to *launches.
bool plan_slot(const pe_graph* g, int64_t K, uint32_t flags, bool times, Plan* p);
int launch_slot(const pe_graph* g, const Plan& p, bool by_pos, int64_t K, const uint8_t* assign, const uint16_t* order,
                uint32_t flags, const pe_outputs& out, void* workspace, cudaStream_t stream, int64_t* launches);

// pe_eval_lane_kernel (plan variant GLOBAL over the compact encoding; state in `gstate`).
int launch_lane(const pe_graph* g, const Plan& p, bool by_pos, int64_t K, const uint8_t* assign, const uint16_t* order,
                uint32_t flags, const pe_outputs& out, uint32_t* gstate, unsigned grid, cudaStream_t stream);

// pe_eval_warp2_kernel (plan variant WARP over the compact encoding).
int launch_warp2(const pe_graph* g, const Plan& p, bool by_pos, int64_t K, const uint8_t* assign, const uint16_t* order,
                 uint32_t flags, const pe_outputs& out, unsigned grid, cudaStream_t stream);

// pe_eval_team_kernel (plan variant TEAM: one block of plan.threads / 32 warps per candidate).
// Adds the number of kernels it launched to *launches.
int launch_team(const pe_graph* g, const Plan& p, bool by_pos, int64_t K, const uint8_t* assign, const uint16_t* order,
                uint32_t flags, const pe_outputs& out, void* workspace, cudaStream_t stream, int64_t* launches);

}  // namespace pe
