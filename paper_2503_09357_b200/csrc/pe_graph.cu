// Host side of the library: description checks, by-predecessor CSR, upload, teardown.
#include <algorithm>
#include <climits>
#include <cstdlib>
#include <cstring>
#include <exception>
#include <memory>
#include <vector>

#include "pe_device.cuh"
#include "pe_graph.h"

namespace {

inline uint32_t align16(uint64_t x) { return (uint32_t)((x + 15u) & ~(uint64_t)15u); }

// Ranges, acyclicity and overflow bounds; fills the bounds when asked.
int check_desc(const pe_graph_desc* d, int64_t* time_bound, int64_t* mem_bound, int32_t* max_indeg, int32_t* levels) {
  if (!d) return PE_ERR_INVALID_ARG;
  const int32_t V = d->num_ops, E = d->num_edges, D = d->num_devices, L = d->num_link_classes;
  if (V < 1 || E < 0 || D < 1 || D > 255 || L < 1 || L > 254) return PE_ERR_INVALID_ARG;
  if (!d->dur || (E > 0 && (!d->edge_src || !d->edge_dst))) return PE_ERR_INVALID_ARG;
  if ((int64_t)E * L > (int64_t)INT32_MAX) return PE_ERR_INVALID_ARG;

  int64_t tsum = 0, msum = 0;
  for (int32_t i = 0; i < V; ++i) {
    if (d->dur[i] < 0) return PE_ERR_RANGE;
    int64_t longest = d->dur[i];
    if (d->dur_by_machine) {   // heterogeneous machines: the bound takes the slowest machine
      longest = 0;
      for (int32_t j = 0; j < D; ++j) {
        const int32_t t = d->dur_by_machine[(size_t)i * D + j];
        if (t < 0) return PE_ERR_RANGE;
        if (t > longest) longest = t;
      }
    }
    tsum += longest;
    if (d->mem_delta) msum += d->mem_delta[i] < 0 ? -(int64_t)d->mem_delta[i] : (int64_t)d->mem_delta[i];
    if (d->mem_weight) {
      if (d->mem_weight[i] < 0) return PE_ERR_RANGE;
      msum += d->mem_weight[i];
    }
  }
  std::vector<int32_t> indeg(V, 0), succ_ptr(V + 1, 0);
  for (int32_t b = 0; b < E; ++b) {
    const int32_t p = d->edge_src[b], i = d->edge_dst[b];
    if (p < 0 || p >= V || i < 0 || i >= V) return PE_ERR_RANGE;
    if (p == i) return PE_ERR_CYCLE;
    indeg[i]++;
    succ_ptr[p + 1]++;
    if (d->comm) {
      int32_t mx = 0;
      for (int32_t l = 0; l < L; ++l) {
        const int32_t cst = d->comm[(size_t)b * L + l];
        if (cst < 0) return PE_ERR_RANGE;
        if (cst > mx) mx = cst;
      }
      tsum += mx;
    }
  }
  if (d->link_class)
    for (int32_t a = 0; a < D * D; ++a)
      if (d->link_class[a] != 0xFF && d->link_class[a] >= L) return PE_ERR_RANGE;
  if (tsum > (int64_t)INT32_MAX || msum > (int64_t)INT32_MAX) return PE_ERR_OVERFLOW;

  // acyclic iff Kahn's algorithm removes every operator
  int32_t mdeg = 0;
  for (int32_t i = 0; i < V; ++i) {
    succ_ptr[i + 1] += succ_ptr[i];
    if (indeg[i] > mdeg) mdeg = indeg[i];
  }
  std::vector<int32_t> succ(E), fill(succ_ptr.begin(), succ_ptr.end() - 1), deg(indeg), stack;
  for (int32_t b = 0; b < E; ++b) succ[fill[d->edge_src[b]]++] = d->edge_dst[b];
  for (int32_t i = 0; i < V; ++i)
    if (deg[i] == 0) stack.push_back(i);
  std::vector<int32_t> level(V, 1);
  int32_t removed = 0, deepest = 1;
  while (!stack.empty()) {
    const int32_t i = stack.back();
    stack.pop_back();
    ++removed;
    if (level[i] > deepest) deepest = level[i];
    for (int32_t q = succ_ptr[i]; q < succ_ptr[i + 1]; ++q) {
      if (level[succ[q]] <= level[i]) level[succ[q]] = level[i] + 1;
      if (--deg[succ[q]] == 0) stack.push_back(succ[q]);
    }
  }
  if (removed != V) return PE_ERR_CYCLE;

  if (time_bound) *time_bound = tsum;
  if (mem_bound) *mem_bound = msum;
  if (max_indeg) *max_indeg = mdeg;
  if (levels) *levels = deepest;
  return PE_OK;
}

// Ancestors of every operator as rows of bits, and a topological order that follows a chain of operators to its end.
struct Ancestors {
  size_t words = 0;
  std::vector<uint64_t> bits;
  std::vector<int32_t> sptr, succ, order;   // successors (with repetitions) in CSR form
  bool of(int32_t i, int32_t a) const { return bits[(size_t)i * words + (size_t)(a / 64)] >> (a % 64) & 1u; }
};
Ancestors find_ancestors(int32_t V, const PeOpRec* ops, const int32_t* pred) {
  Ancestors a;
  a.words = ((size_t)V + 63) / 64;
  a.bits.assign((size_t)V * a.words, 0);
  a.sptr.assign(V + 1, 0);
  const int32_t E = ops[V - 1].edge_begin + ops[V - 1].indeg;
  for (int32_t q = 0; q < E; ++q) a.sptr[pred[q] + 1]++;
  for (int32_t i = 0; i < V; ++i) a.sptr[i + 1] += a.sptr[i];
  a.succ.resize(E);
  std::vector<int32_t> fill(a.sptr.begin(), a.sptr.end() - 1), deg(V), stack;
  for (int32_t i = 0; i < V; ++i)
    for (int32_t q = ops[i].edge_begin; q < ops[i].edge_begin + ops[i].indeg; ++q) a.succ[fill[pred[q]]++] = i;
  for (int32_t i = V - 1; i >= 0; --i) {
    deg[i] = ops[i].indeg;
    if (deg[i] == 0) stack.push_back(i);
  }
  while (!stack.empty()) {
    const int32_t s = stack.back();
    stack.pop_back();
    a.order.push_back(s);
    uint64_t* row = a.bits.data() + (size_t)s * a.words;
    for (int32_t q = ops[s].edge_begin; q < ops[s].edge_begin + ops[s].indeg; ++q) {
      const uint64_t* b = a.bits.data() + (size_t)pred[q] * a.words;
      for (size_t w = 0; w < a.words; ++w) row[w] |= b[w];
      row[pred[q] / 64] |= 1ull << (pred[q] % 64);
    }
    for (int32_t q = a.sptr[s]; q < a.sptr[s + 1]; ++q)
      if (--deg[a.succ[q]] == 0) stack.push_back(a.succ[q]);
  }
  return a;
}

// Chains (of operators each of which is an ancestor of the next) that cover all operators: at most as many operators are
// available at once.  -1 when more than `most` are needed.
int32_t cover_by_chains(const Ancestors& anc, const PeOpRec* ops, const int32_t* pred, int32_t most) {
  std::vector<int32_t> tail, chain(anc.order.size(), -1);
  for (const int32_t s : anc.order) {
    int32_t take = -1;
    for (int32_t q = ops[s].edge_begin; q < ops[s].edge_begin + ops[s].indeg && take < 0; ++q)
      if (tail[chain[pred[q]]] == pred[q]) take = chain[pred[q]];
    for (int32_t t = 0; t < (int32_t)tail.size() && take < 0; ++t)
      if (anc.of(s, tail[t])) take = t;
    if (take < 0) {
      if ((int32_t)tail.size() == most) return -1;
      take = (int32_t)tail.size();
      tail.push_back(s);
    }
    tail[take] = s;
    chain[s] = take;
  }
  return (int32_t)tail.size();
}

// Slots for the slot encoding: operator s takes over the slot of operator p when all successors of p are s or ancestors of
// s (their readings are over in every topological order by then); preferably that of one of its predecessors.  version[s]:
// operators of its slot up to and including s, at most `longest`.  marks: an operator without successors leaves a mark in the
// slot of a predecessor (version 0; one mark a holder) where one is free to take it.  Returns the number of slots, or -1 when
// more than `most` are needed.
int32_t share_slots(const Ancestors& anc, const PeOpRec* ops, const int32_t* pred, int32_t most, int32_t longest, bool marks,
                    std::vector<int32_t>* slot, std::vector<int32_t>* version) {
  const std::vector<int32_t>&sptr = anc.sptr, &succ = anc.succ;
  const int32_t V = (int32_t)anc.order.size();
  slot->assign(V, -1);
  version->assign(V, 0);
  std::vector<int32_t> tail;              // last operator of every slot
  std::vector<int32_t> unread(V), idle;   // successors of an operator still to come; slots whose tail has none
  std::vector<uint8_t> marked(V, 0);
  for (int32_t i = 0; i < V; ++i) unread[i] = sptr[i + 1] - sptr[i];
  for (const int32_t s : anc.order) {
    const int32_t first = ops[s].edge_begin, last = ops[s].edge_begin + ops[s].indeg;
    if (marks && sptr[s] == sptr[s + 1]) {
      for (int32_t q = first; q < last && (*slot)[s] < 0; ++q)
        if (!marked[pred[q]]) { marked[pred[q]] = 1; (*slot)[s] = (*slot)[pred[q]]; }
      if ((*slot)[s] >= 0) continue;   // (its predecessor has a successor that is nobody's ancestor: the slot stays with it)
    }
    auto free_for_s = [&](int32_t t) {   // every successor of the slot's tail is s or an ancestor of s
      const int32_t p = tail[t];
      if ((*version)[p] == longest || sptr[p] == sptr[p + 1]) return false;
      for (int32_t q = sptr[p]; q < sptr[p + 1]; ++q)
        if (succ[q] != s && !anc.of(s, succ[q])) return false;
      return true;
    };
    int32_t take = -1;
    for (int32_t q = first; q < last && take < 0; ++q)
      if (tail[(*slot)[pred[q]]] == pred[q] && free_for_s((*slot)[pred[q]])) take = (*slot)[pred[q]];
    for (size_t t = 0; t < idle.size() && take < 0; ++t)
      if (free_for_s(idle[t])) {
        take = idle[t];
        idle.erase(idle.begin() + (std::ptrdiff_t)t);
      }
    if (take < 0) {
      if ((int32_t)tail.size() == most) return -1;
      take = (int32_t)tail.size();
      tail.push_back(s);
      (*version)[s] = 1;
    } else {
      (*version)[s] = (*version)[tail[take]] + 1;
      tail[take] = s;
    }
    (*slot)[s] = take;
    for (int32_t q = first; q < last; ++q)
      if (--unread[pred[q]] == 0 && tail[(*slot)[pred[q]]] == pred[q]) idle.push_back((*slot)[pred[q]]);
  }
  return (int32_t)tail.size();
}

std::vector<cudaEvent_t*> team_events(pe_graph* g) {
  return {&g->team_fork,    &g->team_join[0], &g->team_join[1], &g->team_join[2], &g->team_in[0],
          &g->team_in[1],   &g->team_done[0], &g->team_done[1], &g->team_back[0], &g->team_back[1]};
}

int create(const pe_graph_desc* d, int cuda_device, pe_graph** out) {
  int64_t tb = 0, mb = 0;
  int32_t mdeg = 0, levels = 1;
  const int rc = check_desc(d, &tb, &mb, &mdeg, &levels);
  if (rc != PE_OK) return rc;
  const int32_t V = d->num_ops, E = d->num_edges, D = d->num_devices, L = d->num_link_classes;

  std::unique_ptr<pe_graph> owner(new pe_graph());
  pe_graph* const g = owner.get();
  g->V = V; g->E = E; g->D = D; g->L = L;
  g->device = cuda_device;
  g->has_weight = d->mem_weight != nullptr;
  g->hetero = d->dur_by_machine != nullptr;
  g->time_bound = tb; g->mem_bound = mb; g->max_indeg = mdeg; g->levels = levels;
  g->d_blob = nullptr; g->d_error = nullptr;

  PeBlobLayout& lay = g->lay;
  uint64_t at = 0;
  lay.ops = (uint32_t)at;    at = align16(at + (uint64_t)V * sizeof(PeOpRec));
  lay.pred = (uint32_t)at;   at = align16(at + (uint64_t)E * 4);
  lay.comm = (uint32_t)at;   at = align16(at + (uint64_t)E * L * 4);
  lay.weight = (uint32_t)at; at = align16(at + (g->has_weight ? (uint64_t)V * 4 : 0));
  lay.cls = (uint32_t)at;    at = align16(at + (uint64_t)D * D);
  lay.cap = (uint32_t)at;    at = align16(at + (uint64_t)D * 4);
  lay.durm = (uint32_t)at;   at = align16(at + (g->hetero ? (uint64_t)V * D * 4 : 0));
  if (at > 0x7FFFFFF0ull) return PE_ERR_INVALID_ARG;
  lay.bytes = (uint32_t)at;

  // by-predecessor CSR: incoming edges of operator i occupy slots edge_begin .. edge_begin + indeg
  std::vector<uint8_t> blob(lay.bytes, 0);
  PeOpRec* ops = (PeOpRec*)(blob.data() + lay.ops);
  int32_t* pred = (int32_t*)(blob.data() + lay.pred);
  int32_t* comm = (int32_t*)(blob.data() + lay.comm);
  for (int32_t i = 0; i < V; ++i) {
    ops[i].indeg = 0;
    ops[i].dur = d->dur[i];
    ops[i].mem_delta = d->mem_delta ? d->mem_delta[i] : 0;
  }
  for (int32_t b = 0; b < E; ++b) ops[d->edge_dst[b]].indeg++;
  int32_t run = 0;
  for (int32_t i = 0; i < V; ++i) { ops[i].edge_begin = run; run += ops[i].indeg; }
  {
    std::vector<int32_t> fill(V);
    for (int32_t i = 0; i < V; ++i) fill[i] = ops[i].edge_begin;
    for (int32_t b = 0; b < E; ++b) {
      const int32_t q = fill[d->edge_dst[b]]++;
      pred[q] = d->edge_src[b];
      for (int32_t l = 0; l < L; ++l) comm[(size_t)q * L + l] = d->comm ? d->comm[(size_t)b * L + l] : 0;
    }
  }
  if (g->has_weight) std::memcpy(blob.data() + lay.weight, d->mem_weight, (size_t)V * 4);
  if (d->link_class) std::memcpy(blob.data() + lay.cls, d->link_class, (size_t)D * D);
  if (g->hetero) std::memcpy(blob.data() + lay.durm, d->dur_by_machine, (size_t)V * D * 4);
  int32_t* cap = (int32_t*)(blob.data() + lay.cap);
  for (int32_t j = 0; j < D; ++j) cap[j] = d->mem_capacity ? d->mem_capacity[j] : INT32_MAX;

  // compact encoding, when every value fits its field
  bool no_channel = false;
  if (d->link_class)
    for (int32_t a = 0; a < D * D; ++a) no_channel = no_channel || d->link_class[a] == 0xFF;
  bool narrow = V <= 65535 && L <= 2 && mdeg <= 255 && E < (1 << 24) && !g->hetero;   // (the compact record has one duration)
  for (int32_t i = 0; narrow && i < V; ++i)
    narrow = ops[i].dur <= 65535 && ops[i].mem_delta >= -128 && ops[i].mem_delta <= 127;
  for (int64_t q = 0; narrow && q < (int64_t)E * L; ++q) narrow = comm[q] <= 65535;
  std::vector<uint8_t> nblob;
  g->narrow_ok = narrow;
  g->d_nblob = nullptr;
  std::memset(&g->nview, 0, sizeof(g->nview));
  if (narrow) {
    PeNarrowView& nv = g->nview;
    nv.V = V; nv.E = E; nv.D = D; nv.L = L;
    nv.has_weight = g->has_weight ? 1 : 0;
    nv.need_cls = (L > 1 || no_channel) ? 1 : 0;
    nv.max_indeg = mdeg;
    uint64_t nat = 0;
    nv.ops = (uint32_t)nat;    nat = align16(nat + (uint64_t)V * 16);
    nv.edges = (uint32_t)nat;  nat = align16(nat + (uint64_t)E * 4 * L);
    nv.weight = (uint32_t)nat; nat = align16(nat + (g->has_weight ? (uint64_t)V * 4 : 0));
    nv.cls = (uint32_t)nat;    nat = align16(nat + (uint64_t)D * D);
    nv.cap = (uint32_t)nat;    nat = align16(nat + (uint64_t)D * 4);
    nv.bytes = (uint32_t)nat;
    nblob.assign(nv.bytes, 0);
    uint32_t* nops = (uint32_t*)(nblob.data() + nv.ops);
    uint32_t* nedges = (uint32_t*)(nblob.data() + nv.edges);
    for (int32_t q = 0; q < E; ++q) {
      const uint32_t lo = ((uint32_t)comm[(size_t)q * L] << 16) | (uint32_t)pred[q];
      if (L == 1) nedges[q] = lo;
      else { nedges[2 * (size_t)q] = lo; nedges[2 * (size_t)q + 1] = (uint32_t)comm[(size_t)q * L + 1]; }
    }
    for (int32_t i = 0; i < V; ++i) {
      uint32_t* r = nops + 4 * (size_t)i;
      const int32_t b = ops[i].edge_begin, n = ops[i].indeg;
      r[1] = ((uint32_t)n << 24) | ((uint32_t)(uint8_t)(int8_t)ops[i].mem_delta << 16) | (uint32_t)ops[i].dur;
      // a missing inline edge points at the sentinel operator V (always "ended at 0", zero delay)
      const uint32_t none = (uint32_t)V;
      if (L == 1) {
        r[2] = n > 0 ? nedges[b] : none;
        r[3] = n > 1 ? nedges[b + 1] : none;
        r[0] = n > 3 ? (uint32_t)b : (n > 2 ? nedges[b + 2] : none);
      } else {
        r[2] = n > 0 ? nedges[2 * (size_t)b] : none;
        r[3] = n > 0 ? nedges[2 * (size_t)b + 1] : 0u;
        r[0] = (uint32_t)b;
      }
    }
    if (g->has_weight) std::memcpy(nblob.data() + nv.weight, d->mem_weight, (size_t)V * 4);
    if (d->link_class) std::memcpy(nblob.data() + nv.cls, d->link_class, (size_t)D * D);
    std::memcpy(nblob.data() + nv.cap, cap, (size_t)D * 4);
  }

  // tile encoding
  bool tile = V <= 65535 && L <= 2 && mdeg <= 255;
  for (int32_t i = 0; tile && i < V; ++i)
    tile = ops[i].dur <= 65535 && ops[i].mem_delta >= -128 && ops[i].mem_delta <= 127;
  for (int64_t q = 0; tile && q < (int64_t)E * L; ++q) tile = comm[q] <= 65535;
  if (g->hetero)
    for (int64_t q = 0; tile && q < (int64_t)V * D; ++q) tile = d->dur_by_machine[q] <= 65535;
  std::vector<uint8_t> tblob;
  g->tile_ok = tile;
  g->d_tblob = nullptr;
  std::memset(&g->tview, 0, sizeof(g->tview));
  if (tile) {
    PeTileView& tv = g->tview;
    tv.V = V; tv.D = D;
    tv.has_weight = g->has_weight ? 1 : 0;
    tv.max_indeg = mdeg;
    bool cut = false;   // some pair of different machines has no channel
    if (d->link_class)
      for (int32_t a = 0; a < D * D; ++a) cut = cut || (d->link_class[a] == 0xFF && a / D != a % D);
    tv.cls_kind = !cut && L == 1 ? 0 : (!cut && D <= 32 ? 2 : 1);
    const bool listed = tv.cls_kind == 0 ? mdeg > 3 : mdeg > 2;
    tv.list_edges = listed ? E : 0;
    uint64_t tat = 0;
    tv.ops = (uint32_t)tat;     tat = align16(tat + (uint64_t)(V + 1) * 16);
    tv.edges = (uint32_t)tat;   tat = align16(tat + (listed ? (uint64_t)E * (tv.cls_kind == 0 ? 4 : 8) : 0));
    tv.slot = (uint32_t)tat;    tat = align16(tat + (listed && tv.cls_kind != 0 ? (uint64_t)V * 4 : 0));
    tv.cls = (uint32_t)tat;     tat = align16(tat + (tv.cls_kind == 1 ? (uint64_t)D * D : 0));
    tv.cls_row = (uint32_t)tat; tat = align16(tat + (tv.cls_kind == 2 ? (uint64_t)D * 4 : 0));
    tv.weight = (uint32_t)tat;  tat = align16(tat + (g->has_weight ? (uint64_t)V * 4 : 0));
    tv.cap = (uint32_t)tat;     tat = align16(tat + (uint64_t)D * 4);
    tv.durm = (uint32_t)tat;    tat = align16(tat + (g->hetero ? (uint64_t)(V + 1) * D * 2 : 0));
    tv.bytes = (uint32_t)tat;
    tblob.assign(tv.bytes, 0);
    uint32_t* r = (uint32_t*)(tblob.data() + tv.ops);
    const uint32_t none = (uint32_t)V;
    auto delays = [&](int32_t q) {   // both classes of CSR edge q
      const uint32_t c0 = (uint32_t)comm[(size_t)q * L];
      return c0 | (L == 2 ? (uint32_t)comm[(size_t)q * L + 1] : c0) << 16;
    };
    for (int32_t i = 0; i <= V; ++i, r += 4) {
      const int32_t b = i < V ? ops[i].edge_begin : 0, n = i < V ? ops[i].indeg : 0;
      r[0] = i < V ? (uint32_t)(uint8_t)(int8_t)ops[i].mem_delta << 24 | (uint32_t)n << 16 | (uint32_t)(g->hetero ? 0 : ops[i].dur) : 0u;
      if (tv.cls_kind == 0) {
        auto edge = [&](int32_t q) { return (uint32_t)comm[q] << 16 | (uint32_t)pred[q]; };
        r[1] = n > 0 ? edge(b) : none;
        r[2] = n > 1 ? edge(b + 1) : none;
        r[3] = n > 3 ? (uint32_t)b : (n > 2 ? edge(b + 2) : none);
      } else {
        r[1] = (n > 0 ? (uint32_t)pred[b] : none) | (n > 1 ? (uint32_t)pred[b + 1] : none) << 16;
        r[2] = n > 0 ? delays(b) : 0u;
        r[3] = n > 1 ? delays(b + 1) : 0u;
      }
    }
    if (listed) {
      uint32_t* te = (uint32_t*)(tblob.data() + tv.edges);
      for (int32_t q = 0; q < E; ++q) {
        if (tv.cls_kind == 0) te[q] = (uint32_t)comm[q] << 16 | (uint32_t)pred[q];
        else { te[2 * (size_t)q] = (uint32_t)pred[q]; te[2 * (size_t)q + 1] = delays(q); }
      }
      if (tv.cls_kind != 0)
        for (int32_t i = 0; i < V; ++i) ((uint32_t*)(tblob.data() + tv.slot))[i] = (uint32_t)ops[i].edge_begin;
    }
    if (tv.cls_kind == 1 && d->link_class) std::memcpy(tblob.data() + tv.cls, d->link_class, (size_t)D * D);
    if (tv.cls_kind == 2 && d->link_class)
      for (int32_t j = 0; j < D; ++j)
        for (int32_t x = 0; x < D; ++x)
          if (x != j && d->link_class[(size_t)x * D + j] == 1) ((uint32_t*)(tblob.data() + tv.cls_row))[j] |= 1u << x;
    if (g->has_weight) std::memcpy(tblob.data() + tv.weight, d->mem_weight, (size_t)V * 4);
    std::memcpy(tblob.data() + tv.cap, cap, (size_t)D * 4);
    if (g->hetero)
      for (int64_t q = 0; q < (int64_t)V * D; ++q) ((uint16_t*)(tblob.data() + tv.durm))[q] = (uint16_t)d->dur_by_machine[q];
  }

  Ancestors anc;   // (dense graphs that no encoding below serves take as long to find them as for all the rest)
  auto ancestors = [&]() -> const Ancestors& {
    if (anc.words == 0) anc = find_ancestors(V, ops, pred);
    return anc;
  };

  // slot encoding
  std::vector<uint8_t> sblob;
  g->slot_ok = false;
  g->d_sblob = nullptr;
  std::memset(&g->sview, 0, sizeof(g->sview));
  int64_t asum = 0;
  int32_t longest_field = 1;   // of the durations and delays
  for (int32_t i = 0; i < V; ++i) {
    asum += std::abs((int64_t)ops[i].mem_delta);
    for (int32_t j = 0; j < (g->hetero ? D : 1); ++j)
      longest_field = std::max(longest_field, g->hetero ? d->dur_by_machine[(size_t)i * D + j] : ops[i].dur);
  }
  for (int64_t q = 0; q < (int64_t)E * L; ++q) longest_field = std::max(longest_field, comm[q]);
  int vbits = 8;
  while (vbits > 0 && (tb >= (int64_t)1 << (24 - vbits) || (int64_t)longest_field << vbits > 65535)) --vbits;
  if (tile && V <= 4096 && asum < 32768 && vbits >= 4) {
    std::vector<int32_t> slot, version;
    bool marks = false;
    int32_t n = share_slots(ancestors(), ops, pred, V / 4, (1 << (vbits - 1)) - 1, false, &slot, &version);
    if (n < 0 && g->tview.cls_kind == 0 && mdeg <= 3) {
      marks = true;
      n = share_slots(anc, ops, pred, (int32_t)(0.65 * V), (1 << (vbits - 2)) - 1, true, &slot, &version);
    }
    if (n >= 0) {
      g->slot_ok = true;
      PeSlotView& sv = g->sview;
      sv.V = V; sv.E = E; sv.D = D; sv.nslots = n;
      sv.has_weight = g->has_weight ? 1 : 0;
      sv.cls_kind = g->tview.cls_kind;
      sv.vbits = vbits;
      sv.marks = marks ? 1 : 0;
      struct Source { uint32_t slot, c0, c1; };   // delays << vbits | version, per class
      std::vector<std::vector<Source>> sources(V + 1);
      std::vector<uint8_t> own_first(V + 1, 0);
      sv.max_sources = 0;
      for (int32_t i = 0; i < V; ++i) {
        const uint32_t before = (uint32_t)version[i] - 1u;
        bool chained = false;
        for (int32_t q = ops[i].edge_begin; q < ops[i].edge_begin + ops[i].indeg; ++q)
          chained = chained || (slot[pred[q]] == slot[i] && version[pred[q]] == version[i] - 1);
        if (!chained && !marks) { sources[i].push_back({(uint32_t)slot[i], before, before}); own_first[i] = 1; }
        for (int32_t q = ops[i].edge_begin; q < ops[i].edge_begin + ops[i].indeg; ++q) {
          const uint32_t v = (uint32_t)version[pred[q]], c0 = (uint32_t)comm[(size_t)q * L], c1 = L == 2 ? (uint32_t)comm[(size_t)q * L + 1] : c0;
          sources[i].push_back({(uint32_t)slot[pred[q]], c0 << vbits | v, c1 << vbits | v});
        }
        sv.max_sources = std::max(sv.max_sources, (int32_t)sources[i].size());
      }
      std::vector<uint32_t> list, list_at(V + 1, 0), rec((size_t)(V + 1) * 4, 0);
      const bool padded = sv.max_sources <= 8;   // six places an operator, places without a source name row nslots
      const Source none = {(uint32_t)n, 0u, 0u};
      auto add_list = [&](const std::vector<Source>& src, size_t from) {
        const size_t count = padded ? 6 : src.size() - from;
        for (size_t q = 0; q < count; ++q) {
          const Source& x = from + q < src.size() ? src[from + q] : none;
          const uint32_t mark = q + 1 == count ? 0x1000u : 0u;
          if (sv.cls_kind == 0) list.push_back(x.c0 << 16 | mark | x.slot);
          else { list.push_back(mark | x.slot); list.push_back(x.c0 | x.c1 << 16); }
        }
        while (padded && list.size() % 4 != 0) list.push_back((uint32_t)n);
      };
      for (int32_t i = 0; i <= V; ++i) {   // (record V stands for entries that are no operator)
        uint32_t* r = rec.data() + 4 * (size_t)i;
        const std::vector<Source>& src = sources[i];
        const uint32_t own = i < V ? (uint32_t)slot[i] : (uint32_t)n + 1u;
        auto get = [&](size_t q) { return q < src.size() ? src[q] : none; };
        r[0] = (own & 0xFFu) << 16;
        if (i < V) r[0] |= (uint32_t)(uint8_t)(int8_t)ops[i].mem_delta << 24 | (uint32_t)(g->hetero ? 0 : ops[i].dur) << vbits | (version[i] > 0 ? (uint32_t)version[i] : 1u << (vbits - 1));
        if (sv.cls_kind == 0) {
          auto edge = [&](size_t q) { return get(q).c0 << 16 | get(q).slot; };
          r[1] = edge(0) | (own >> 8) << 12;
          r[2] = edge(1) | (src.size() > 3 ? 0x1000u : 0u) | (own_first[i] ? 0x2000u : 0u);
          r[3] = src.size() > 3 ? (uint32_t)list.size() : edge(2);
          if (src.size() > 3) add_list(src, 2);
        } else {
          r[1] = get(0).slot | (own >> 8) << 12 | get(1).slot << 16 | (src.size() > 2 ? 0x10000000u : 0u) | (own_first[i] ? 0x20000000u : 0u);
          r[2] = get(0).c0 | get(0).c1 << 16;
          r[3] = get(1).c0 | get(1).c1 << 16;
          list_at[i] = (uint32_t)(list.size() / 2);
          if (src.size() > 2) add_list(src, 2);
        }
      }
      std::vector<uint16_t> dur16(V), durm16(g->hetero ? (size_t)(V + 1) * D : 0, 0);
      for (int32_t i = 0; i < V; ++i) dur16[i] = (uint16_t)ops[i].dur;
      if (g->hetero)
        for (size_t q = 0; q < (size_t)V * D; ++q) durm16[q] = (uint16_t)(d->dur_by_machine[q] << vbits);
      auto put = [&](const void* at, size_t bytes) {
        const size_t off = sblob.size();
        sblob.resize(align16(off + bytes), 0);
        if (bytes) std::memcpy(sblob.data() + off, at, bytes);
        return (uint32_t)off;
      };
      sv.ops = put(rec.data(), rec.size() * 4);
      sv.list = put(list.data(), list.size() * 4);
      sv.list_at = put(list_at.data(), list.empty() || sv.cls_kind == 0 ? 0 : list_at.size() * 4);
      sv.cls = put(tblob.data() + g->tview.cls, sv.cls_kind == 1 ? (size_t)D * D : 0);
      sv.cls_row = put(tblob.data() + g->tview.cls_row, sv.cls_kind == 2 ? (size_t)D * 4 : 0);
      sv.cap = put(cap, (size_t)D * 4);
      sv.durm = put(durm16.data(), durm16.size() * 2);
      sv.bytes = (uint32_t)sblob.size();
      sv.dur = put(dur16.data(), (size_t)V * 2);
      sv.weight = put(d->mem_weight, g->has_weight ? (size_t)V * 4 : 0);
      sv.total = (uint32_t)sblob.size();
    }
  }

  // forward view (successor lists) for priority-list decoding
  std::vector<uint8_t> fblob;
  g->fwd_ok = V <= 65536 && mdeg <= 255;
  g->d_fwd = nullptr;
  std::memset(&g->fview, 0, sizeof(g->fview));
  if (g->fwd_ok) {
    PeFwdView& fv = g->fview;
    std::vector<uint32_t> sptr(V + 1, 0);
    for (int32_t b = 0; b < E; ++b) sptr[d->edge_src[b] + 1]++;
    for (int32_t i = 0; i < V; ++i) sptr[i + 1] += sptr[i];
    std::vector<uint16_t> succ(E);
    std::vector<uint32_t> fill(sptr.begin(), sptr.end() - 1);
    for (int32_t b = 0; b < E; ++b) succ[fill[d->edge_src[b]]++] = (uint16_t)d->edge_dst[b];
    std::vector<uint8_t> uindeg(V, 0);
    std::vector<uint32_t> uptr(V + 1, 0);
    std::vector<uint16_t> usucc, more;
    usucc.reserve(E);
    int32_t seven = 0;
    fv.short_lists = 1;
    for (int32_t i = 0; i < V; ++i) {
      std::sort(succ.begin() + sptr[i], succ.begin() + sptr[i + 1]);
      const auto end = std::unique(succ.begin() + sptr[i], succ.begin() + sptr[i + 1]);
      usucc.insert(usucc.end(), succ.begin() + sptr[i], end);
      uptr[i + 1] = (uint32_t)usucc.size();
      const uint32_t n = uptr[i + 1] - uptr[i];
      seven += n > 6 && n <= 14;
      if (n > 255) fv.short_lists = 0;
    }
    fv.rec_bytes = seven > V / 50 ? 32 : 16;
    const uint32_t halves = fv.rec_bytes / 2, inl = halves - 2;
    std::vector<uint16_t> rec((size_t)V * halves, (uint16_t)V);
    for (int32_t i = 0; i < V; ++i) {
      const uint32_t n = uptr[i + 1] - uptr[i];
      uint16_t* r = rec.data() + (size_t)i * halves;
      r[0] = (uint16_t)n;
      for (uint32_t q = 0; q < n; ++q) {
        uindeg[usucc[uptr[i] + q]]++;
        if (n <= inl) r[1 + q] = usucc[uptr[i] + q];
      }
      if (n > inl) {
        r[0] = 64;
        r[1] = (uint16_t)n;
        r[2] = (uint16_t)(more.size() & 0xFFFFu);
        r[3] = (uint16_t)(more.size() >> 16);
        more.insert(more.end(), usucc.begin() + uptr[i], usucc.begin() + uptr[i + 1]);
      }
    }
    fv.V = V; fv.E = (int32_t)usucc.size();
    // pool kernel: joins, roots, successors
    std::vector<uint8_t> pool;
    const int32_t chains = fv.short_lists && V <= 4096 ? cover_by_chains(ancestors(), ops, pred, 32) : -1;
    if (chains >= 0) {
      std::vector<uint32_t> join(V, 0xFFFFu), prec((size_t)V * 2, 0), pmore;
      std::vector<uint8_t> joins;
      std::vector<uint16_t> roots;
      int32_t leaves = 0;
      for (int32_t i = 0; i < V; ++i) {
        if (uindeg[i] > 1) { join[i] = (uint32_t)joins.size(); joins.push_back((uint8_t)(uindeg[i] - 1)); }
        if (uindeg[i] == 0) roots.push_back((uint16_t)i);
      }
      for (int32_t i = 0; i < V; ++i) {
        const uint32_t n = uptr[i + 1] - uptr[i];
        leaves += n == 0 ? 1 : 0;
        auto entry = [&](uint32_t q) { return (uint32_t)usucc[q] | join[usucc[q]] << 16; };
        prec[2 * (size_t)i] = n > 0 ? entry(uptr[i]) : 0u;
        prec[2 * (size_t)i + 1] = n << 24 | (uint32_t)pmore.size();
        for (uint32_t q = 1; q < n; ++q) pmore.push_back(entry(uptr[i] + q));
      }
      fv.num_roots = (int32_t)roots.size(); fv.num_joins = (int32_t)joins.size();
      fv.places = (chains + 7) / 8 * 8;
      fv.turns = (int32_t)usucc.size() + leaves;
      auto put = [&](const void* from, size_t n) {
        const size_t off = pool.size();
        pool.resize(align16(off + n), 0);
        if (n) std::memcpy(pool.data() + off, from, n);
        return (uint32_t)off;
      };
      pmore.push_back(0xFFFF0000u);   // (read, not used, behind the last successor of an operator)
      put(prec.data(), prec.size() * 4);
      fv.pmore = put(pmore.data(), pmore.size() * 4);
      fv.roots = put(roots.data(), roots.size() * 2);
      fv.joins = put(joins.data(), joins.size());
      fv.pool_bytes = (uint32_t)pool.size();
    }
    uint64_t fat = 0;
    fv.ptr = (uint32_t)fat;   fat = align16(fat + (uint64_t)(V + 1) * 4);
    fv.succ = (uint32_t)fat;  fat = align16(fat + (uint64_t)usucc.size() * 2);
    fv.indeg = (uint32_t)fat; fat = align16(fat + (uint64_t)V);
    fv.rec = (uint32_t)fat;   fat = align16(fat + (uint64_t)V * fv.rec_bytes);
    fv.more = (uint32_t)fat;  fat = align16(fat + (uint64_t)more.size() * 2);
    fv.prec = (uint32_t)fat;  fat = align16(fat + pool.size());
    fblob.assign((size_t)fat, 0);
    auto put = [&](uint32_t at, const void* from, size_t n) { if (n) std::memcpy(fblob.data() + at, from, n); };
    put(fv.ptr, uptr.data(), (size_t)(V + 1) * 4);
    put(fv.succ, usucc.data(), usucc.size() * 2);
    put(fv.indeg, uindeg.data(), (size_t)V);
    put(fv.rec, rec.data(), (size_t)V * fv.rec_bytes);
    put(fv.more, more.data(), more.size() * 2);
    put(fv.prec, pool.data(), pool.size());
  }

  // one allocation and one copy for all encodings (each on a 256-byte boundary), the status word last
  std::vector<uint8_t> all;
  auto place = [&](const std::vector<uint8_t>& part) {
    const size_t at = (all.size() + 255) / 256 * 256;
    all.resize(at);
    all.insert(all.end(), part.begin(), part.end());
    return at;
  };
  const size_t at_blob = place(blob), at_n = place(nblob), at_t = place(tblob), at_f = place(fblob), at_s = place(sblob);
  const size_t at_err = place(std::vector<uint8_t>(256, 0));
  int prev = -1, sms = 0, optin = 0, per_sm = 0;
  bool ok = cudaGetDevice(&prev) == cudaSuccess && cudaSetDevice(cuda_device) == cudaSuccess &&
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, cuda_device) == cudaSuccess &&
            cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, cuda_device) == cudaSuccess &&
            cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, cuda_device) == cudaSuccess;
  if (ok) {
    g->sm_count = sms;
    g->smem_optin = (size_t)optin;
    g->smem_per_sm = (size_t)per_sm;
    ok = cudaMalloc((void**)&g->d_blob, all.size()) == cudaSuccess &&
         cudaMemcpy(g->d_blob, all.data(), all.size(), cudaMemcpyHostToDevice) == cudaSuccess;
    if (ok) {
      uint8_t* base = g->d_blob + at_blob;   // (= d_blob: the generic blob comes first)
      g->d_nblob = narrow ? base + at_n : nullptr;
      g->d_tblob = tile ? base + at_t : nullptr;
      g->d_fwd = g->fwd_ok ? base + at_f : nullptr;
      g->d_sblob = g->slot_ok ? base + at_s : nullptr;
      g->d_error = reinterpret_cast<int*>(base + at_err);
    }
    if (ok) {
      ok = cudaStreamCreateWithFlags(&g->copy_in, cudaStreamNonBlocking) == cudaSuccess &&
           cudaStreamCreateWithFlags(&g->copy_out, cudaStreamNonBlocking) == cudaSuccess &&
           cudaEventCreateWithFlags(&g->ev_begin, cudaEventDisableTiming) == cudaSuccess &&
           cudaEventCreateWithFlags(&g->ev_end, cudaEventDisableTiming) == cudaSuccess &&
           cudaStreamCreateWithFlags(&g->team_stream[0], cudaStreamNonBlocking) == cudaSuccess &&
           cudaStreamCreateWithFlags(&g->team_stream[1], cudaStreamNonBlocking) == cudaSuccess;
      int least = 0, greatest = 0;
      ok = ok && cudaDeviceGetStreamPriorityRange(&least, &greatest) == cudaSuccess &&
           cudaStreamCreateWithPriority(&g->team_copy, cudaStreamNonBlocking, greatest) == cudaSuccess;
      for (cudaEvent_t* e : team_events(g)) ok = ok && cudaEventCreateWithFlags(e, cudaEventDisableTiming) == cudaSuccess;
      for (int q = 0; ok && q < pe_graph::kMaxChunks; ++q)
        ok = cudaEventCreateWithFlags(&g->ev_in[q], cudaEventDisableTiming) == cudaSuccess &&
             cudaEventCreateWithFlags(&g->ev_done[q], cudaEventDisableTiming) == cudaSuccess;
    }
  }
  if (prev >= 0) cudaSetDevice(prev);
  if (!ok) {
    cudaGetLastError();
    if (g->d_blob) cudaFree(g->d_blob);
    if (g->copy_in) cudaStreamDestroy(g->copy_in);
    if (g->copy_out) cudaStreamDestroy(g->copy_out);
    if (g->ev_begin) cudaEventDestroy(g->ev_begin);
    if (g->ev_end) cudaEventDestroy(g->ev_end);
    for (cudaStream_t s : {g->team_stream[0], g->team_stream[1], g->team_copy})
      if (s) cudaStreamDestroy(s);
    for (cudaEvent_t* e : team_events(g))
      if (*e) cudaEventDestroy(*e);
    for (int q = 0; q < pe_graph::kMaxChunks; ++q) {
      if (g->ev_in[q]) cudaEventDestroy(g->ev_in[q]);
      if (g->ev_done[q]) cudaEventDestroy(g->ev_done[q]);
    }
    cudaGetLastError();
    return PE_ERR_CUDA;
  }
  *out = owner.release();
  return PE_OK;
}

}  // namespace

extern "C" int pe_graph_validate(const pe_graph_desc* desc) {
  try {
    return check_desc(desc, nullptr, nullptr, nullptr, nullptr);
  } catch (const std::exception&) {   // (no memory for the scratch arrays)
    return PE_ERR_CUDA;
  }
}

extern "C" int pe_graph_create(const pe_graph_desc* d, int cuda_device, pe_graph** out) {
  if (!out) return PE_ERR_INVALID_ARG;
  *out = nullptr;
  try {
    return create(d, cuda_device, out);
  } catch (const std::exception&) {
    return PE_ERR_CUDA;
  }
}

extern "C" int pe_destroy(pe_graph* g) {
  if (!g) return PE_OK;
  int prev = -1;
  cudaGetDevice(&prev);
  cudaSetDevice(g->device);
  cudaStreamDestroy(g->copy_in);
  cudaStreamDestroy(g->copy_out);
  cudaEventDestroy(g->ev_begin);
  cudaEventDestroy(g->ev_end);
  for (cudaStream_t s : {g->team_stream[0], g->team_stream[1], g->team_copy}) cudaStreamDestroy(s);
  for (cudaEvent_t* e : team_events(g)) cudaEventDestroy(*e);
  for (int q = 0; q < pe_graph::kMaxChunks; ++q) { cudaEventDestroy(g->ev_in[q]); cudaEventDestroy(g->ev_done[q]); }
  const bool ok = cudaFree(g->d_blob) == cudaSuccess;
  if (prev >= 0) cudaSetDevice(prev);
  delete g;
  return ok ? PE_OK : PE_ERR_CUDA;
}

extern "C" int pe_graph_poll_error(pe_graph* g, void* cuda_stream) {
  if (!g) return PE_ERR_INVALID_ARG;
  int word = 0;
  if (cudaStreamSynchronize((cudaStream_t)cuda_stream) != cudaSuccess) return PE_ERR_CUDA;
  if (cudaMemcpy(&word, g->d_error, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return PE_ERR_CUDA;
  if (word != 0 && cudaMemset(g->d_error, 0, sizeof(int)) != cudaSuccess) return PE_ERR_CUDA;
  return word;
}

// Self-test of the bounded wait: the barrier is told to expect bytes that no copy will ever bring, so the
// wait runs out after `limit` polls, the error word is set and the block returns - nothing is in flight.
__global__ void pe_selftest_wait_kernel(int* err, int limit) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) pe::mbar_init(&bar, 1);
  __syncthreads();
  if (threadIdx.x == 0) pe::mbar_expect_tx(&bar, 16);
  __syncthreads();
  if (!pe::mbar_wait_bounded(&bar, 0, limit)) atomicExch(err, PE_ERR_TIMEOUT);
}

extern "C" int pe_selftest_wait_timeout(pe_graph* g, void* cuda_stream) {
  if (!g) return PE_ERR_INVALID_ARG;
  int prev = -1;
  if (cudaGetDevice(&prev) != cudaSuccess) return PE_ERR_CUDA;
  if (prev != g->device && cudaSetDevice(g->device) != cudaSuccess) return PE_ERR_CUDA;
  pe_selftest_wait_kernel<<<1, 32, 0, (cudaStream_t)cuda_stream>>>(g->d_error, 1024);
  const int ret = cudaGetLastError() == cudaSuccess ? PE_OK : PE_ERR_CUDA;
  if (prev != g->device) cudaSetDevice(prev);
  return ret;
}

extern "C" const char* pe_strerror(int code) {
  switch (code) {
    case PE_OK: return "ok";
    case PE_ERR_INVALID_ARG: return "invalid argument";
    case PE_ERR_CYCLE: return "operator graph has a cycle";
    case PE_ERR_RANGE: return "value out of range (negative duration/communication/weight, edge endpoint or link class)";
    case PE_ERR_OVERFLOW: return "time or memory bound does not fit in int32";
    case PE_ERR_CUDA: return "CUDA runtime call failed";
    case PE_ERR_WORKSPACE: return "workspace missing or too small";
    case PE_ERR_TIMEOUT: return "bounded device-side wait expired";
    case PE_ERR_UNSUPPORTED: return "kernel variant cannot run this problem size";
    case PE_ERR_SCRATCH_LIMIT: return "batch needs more scratch than the built-in no-allocation array holds";
    default: return "unknown error code";
  }
}
