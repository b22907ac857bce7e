// Internal: host-side graph handle and the device-side view kernels receive.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <mutex>

#include "pe.h"

// One record per operator i, 16 bytes: where its incoming edges start in the by-predecessor
// CSR, how many there are, its duration D^o_i and its memory adjustment A_i.
struct PeOpRec {
  int32_t edge_begin;
  int32_t indeg;
  int32_t dur;
  int32_t mem_delta;
};

// Byte offsets of the arrays inside the graph blob (one contiguous, 16-byte aligned block in
// device memory, copied verbatim into shared memory by the kernels that stage it).
struct PeBlobLayout {
  uint32_t ops;     // PeOpRec[V]
  uint32_t pred;    // int32[E]      predecessor id of CSR slot q
  uint32_t comm;    // int32[E*L]    D^c of CSR slot q over link class l at q*L + l
  uint32_t weight;  // int32[V]      W_i (present only if has_weight)
  uint32_t cls;     // uint8[D*D]    link class of (machine of predecessor, machine of successor)
  uint32_t cap;     // int32[D]      capacity (INT32_MAX where there is no limit)
  uint32_t durm;    // int32[V*D]    duration of operator i on machine j at i*D + j (present only if hetero)
  uint32_t bytes;   // total, multiple of 16
};

// What a kernel needs to know about the graph; `base` points at the blob (global or shared).
struct PeGraphView {
  int32_t V, E, D, L;
  int32_t has_weight;
  int32_t hetero;   // durations depend on the machine (the blob holds durm)
  PeBlobLayout lay;
};

// Compact ("narrow") encoding of the same graph, built when every value fits: V <= 65535,
// D^o and D^c below 65536, A in int8, L <= 2, in-degree <= 255, E < 2^24.  One 16-byte record
// per operator carries its first incoming edges inline, so the common operator needs a single
// load.  An edge is  lo = comm[class 0] << 16 | pred  (plus  hi = comm[class 1]  when L == 2).
//   w1 = indeg << 24 | (uint8)A << 16 | dur
//   L == 1: w2, w3 = lo of incoming edges 0 and 1;
//           w0 = lo of incoming edge 2 when indeg <= 3, else the CSR slot of the first incoming
//           edge (edges 2.. are then read from the CSR list)
//   L == 2: (w2, w3) = (lo, hi) of incoming edge 0; w0 = CSR slot of the first incoming edge
// followed by all incoming edges again in CSR order (4 bytes each for L == 1, 8 for L == 2).
// An inline slot without an edge holds pred = V with zero delay: kernels keep a sentinel state
// row V ("ended at time 0 on machine 0"), so the slot can be evaluated without a branch.
struct PeNarrowView {
  int32_t V, E, D, L;
  int32_t has_weight;
  int32_t need_cls;   // the link-class table must be consulted (L > 1 or some pair has no channel)
  int32_t max_indeg;  // largest in-degree (kernels skip the third inline slot when it is <= 2)
  uint32_t ops;       // uint4[V]
  uint32_t edges;     // uint32[E] (L == 1) or uint2[E] (L == 2)
  uint32_t weight;    // int32[V] if has_weight
  uint32_t cls;       // uint8[D*D]
  uint32_t cap;       // int32[D]
  uint32_t bytes;     // total, multiple of 16
};

// Tile encoding, the one that pe_eval_tile_kernel stages into shared memory (V <= 65535, durations and
// delays below 65536, A in int8, L <= 2, in-degree <= 255; durations by machine allowed).  One 16-byte
// record per operator plus a record for the sentinel operator V:
//   x = (uint8)A << 24 | indeg << 16 | dur
//   one class, every pair connected (cls_kind 0):  y, z, w = incoming edges 0, 1, 2 as delay << 16 | pred;
//     w = slot of the first incoming edge in the edge list when indeg > 3 (edges 2.. are read from there)
//   otherwise:  y = pred 0 | pred 1 << 16,  z, w = delay of edge 0, 1:  class 0 | class 1 << 16;
//     edges 2.. are in the edge list, the first incoming edge of operator i at slot[i]
// Missing edges name the sentinel with zero delay.  The edge list (delay << 16 | pred, or
// {pred, class 0 | class 1 << 16}) is present only if some operator has more edges than a record holds.
struct PeTileView {
  int32_t V, D;
  int32_t has_weight;
  int32_t cls_kind;    // 0: one class, all connected; 1: class table; 2: two classes, all connected, D <= 32: row bits
  int32_t max_indeg;
  int32_t list_edges;  // edges in the list (0 or E)
  uint32_t ops;        // uint4[V + 1]
  uint32_t edges;      // uint32[E] or uint2[E]
  uint32_t slot;       // uint32[V] (class kinds 1 and 2 with an edge list)
  uint32_t cls;        // uint8[D*D] (kind 1)
  uint32_t cls_row;    // uint32[D] (kind 2): bit x of row j = class of the channel x -> j
  uint32_t weight;     // int32[V] if has_weight
  uint32_t cap;        // int32[D]
  uint32_t durm;       // uint16[V*D] duration of operator i on machine j at i*D + j (heterogeneous machines; row V = 0 follows)
  uint32_t bytes;      // total, multiple of 16
};

// Slot encoding, for graphs through which few results are alive at a time (see pe_kernel_slot.cuh): operators share
// `nslots` state words.  Built when the tile encoding exists, V <= 4096, V / 4 slots are enough (with `marks`, for one class
// and at most three incoming edges: 0.65 V), the levels without weights
// stay below 2^15, and durations, delays and the time bound leave `vbits` >= 4 bits for versions: times are kept in units of
// 2^vbits, a field below stands for `value << vbits | version`.  One 16-byte record per operator, and record V for entries
// that are no operator:
//   x = (uint8)A << 24 | own slot (low byte) << 16 | dur, own version;  bits 12..15 of y = own slot >> 8
//   one class, every pair connected (cls_kind 0):  y, z, w = sources 0, 1, 2 as (delay, version) << 16 | slot; bit 12 of z:
//     more than three sources, w = place of source 2 in the list ((delay, version) << 16 | last << 12 | slot); bit 13: see below
//   otherwise:  y = slot 0 | slot 1 << 16 | more than two sources << 28,  z, w = source 0, 1:  (delay, version) of class 0 |
//     of class 1 << 16;  list_at[operator] = place of source 2 in the list ({last << 12 | slot, as z}); bit 29 of y: see below
// Sources are the incoming edges.  An operator whose slot was not held by one of its predecessors has its own slot in front
// of them, with the version of the operator that held it and no delay (that operator is an ancestor, or there was none):
// bit 13 / 29.  With `marks` there are no such sources: every operator reads its own slot besides, and one without successors
// has the slot of a predecessor and the top bit of `version` instead of one.  With at most eight sources an operator's part of the list has six places (eight words or twelve).
// Slot nslots stands for missing sources (it holds "ended at 0", version 0), nslots + 1 is that of entries
// that are no operator (not initialised: their candidate is flagged already).
struct PeSlotView {
  int32_t V, E, D;
  int32_t nslots;
  int32_t vbits;
  int32_t marks;
  int32_t has_weight;
  int32_t cls_kind;    // as in PeTileView
  int32_t max_sources;
  uint32_t ops;        // uint4[V + 1]
  uint32_t list;       // uint32[] or uint2[]
  uint32_t list_at;    // uint32[V + 1] (class kinds 1 and 2 with a list)
  uint32_t cls;        // uint8[D*D] (kind 1)
  uint32_t cls_row;    // uint32[D] (kind 2)
  uint32_t cap;        // int32[D]
  uint32_t durm;       // uint16[(V + 1)*D], << vbits (heterogeneous machines)
  uint32_t bytes;      // of the arrays above, which the recurrence keeps in shared memory; multiple of 16
  uint32_t dur;        // uint16[V]
  uint32_t weight;     // int32[V] if has_weight
  uint32_t total;      // multiple of 16
};

// Forward view of the DAG for priority-list decoding, built when V <= 65536 and no operator has more than
// 255 incoming edges.  Parallel edges count once (a predecessor is placed once).  One record per operator of
// rec_bytes / 2 uint16: {n, successors 0 .. inl - 1, V} with inl = rec_bytes / 2 - 2, places without a successor hold V;
// with n > inl: {64, n, first entry in `more` as two halves, ...}, all n successors in `more`.  ptr / succ hold the
// same lists in CSR form.
struct PeFwdView {
  int32_t V, E;    // E: edges without repetitions
  uint32_t ptr;    // uint32[V + 1]
  uint32_t succ;   // uint16[E]
  uint32_t indeg;  // uint8[V]
  uint32_t rec;    // uint16[V][rec_bytes / 2]
  uint32_t rec_bytes;   // 16, or 32 where a fiftieth of the operators has 7 to 14 successors
  uint32_t more;   // uint16[]
  int32_t short_lists;  // no operator has more than 255 successors
  // For pe_decode_pool_kernel (pool_bytes 0: absent; V <= 4096, at most 32 chains cover all operators, at most 255 successors
  // an operator); offsets below count from
  // prec, one block that is copied to shared memory.  A successor is operator | its place among the joins << 16 (0xFFFF: it has
  // one predecessor); prec: {first successor, how many << 24 | the others' place in pmore}.
  int32_t num_roots, num_joins;
  int32_t places;       // of the pool: chains that cover the operators, a multiple of 8
  int32_t turns;        // of the kernel's loop: successors, and operators without one
  uint32_t prec;        // uint2[V]
  uint32_t pmore;       // uint32[]
  uint32_t roots;       // uint16[num_roots]
  uint32_t joins;       // uint8[num_joins]: predecessors less one
  uint32_t pool_bytes;  // multiple of 16
};

struct pe_graph {
  int32_t V, E, D, L;
  int device;
  bool has_weight;
  bool hetero;         // durations depend on the machine
  int64_t time_bound;  // sum dur + sum_e max_l comm: no start/end time exceeds it
  int64_t mem_bound;   // sum |A| + sum W
  int32_t max_indeg;
  int32_t levels;      // operators on the longest path
  PeBlobLayout lay;
  uint8_t* d_blob;     // device copy of the blob; one allocation that also holds the encodings below and d_error
  bool narrow_ok;      // the compact encoding exists
  PeNarrowView nview;
  uint8_t* d_nblob;    // device copy of the compact encoding (nullptr if !narrow_ok)
  bool tile_ok;        // the tile encoding exists
  PeTileView tview;
  uint8_t* d_tblob;    // device copy of the tile encoding (nullptr if !tile_ok)
  bool slot_ok;        // the slot encoding exists
  PeSlotView sview;
  uint8_t* d_sblob;    // device copy of the slot encoding (nullptr if !slot_ok)
  bool fwd_ok;         // the forward view exists
  PeFwdView fview;
  uint8_t* d_fwd;      // device copy of the forward view (nullptr if !fwd_ok)
  int* d_error;        // device status word (0 = ok)
  // pe_eval_batch_host pipelines copies and kernels over candidate chunks: one stream per copy
  // direction and one event per chunk and stage, created with the graph; `host_mutex` serialises
  // host-buffer calls on the same graph because they share these.
  static constexpr int kMaxChunks = 16;
  cudaStream_t copy_in, copy_out;
  cudaEvent_t ev_begin, ev_end, ev_in[kMaxChunks], ev_done[kMaxChunks];
  std::mutex host_mutex;
  // pe_eval_batch with the TEAM variant works through chunks of candidates: evaluations alternate between two side
  // streams, the staging transpositions have a third one of higher priority, so that those of one chunk overlap the
  // evaluation of another.  `team_mutex` serialises the enqueueing of such calls on one graph (they share the events).
  cudaStream_t team_stream[2], team_copy;
  cudaEvent_t team_fork, team_join[3], team_in[2], team_done[2], team_back[2];
  std::mutex team_mutex;
  int sm_count;
  size_t smem_optin;   // max dynamic shared memory per block
  size_t smem_per_sm;  // shared memory of an SM
};

inline PeGraphView pe_view(const pe_graph* g) {
  PeGraphView v;
  v.V = g->V; v.E = g->E; v.D = g->D; v.L = g->L;
  v.has_weight = g->has_weight ? 1 : 0;
  v.hetero = g->hetero ? 1 : 0;
  v.lay = g->lay;
  return v;
}
