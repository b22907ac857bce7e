// Launcher of pe_eval_team_kernel (instantiated in pe_team_nw*.cu), with the staging transpositions around it.
#include "pe_team_launch.h"
#include "pe_transpose.cuh"

#include <mutex>

namespace pe {

namespace {

template <bool BY_POS>
int launch1(const TeamCall& t) {
  switch (t.p->threads / 32) {
    case 2: return launch_team_nw2(t, BY_POS);
    case 4: return launch_team_nw4(t, BY_POS);
    case 6: return launch_team_nw6(t, BY_POS);
    default: return PE_ERR_UNSUPPORTED;
  }
}

// out[C][out_ld] = transposed in[R][in_ld] (element size S)
template <int S>
void transpose(const void* in, void* out, int64_t R, int64_t C, int64_t in_ld, int64_t out_ld, cudaStream_t stream) {
  constexpr int TR = 32 * (4 / S);
  const dim3 grid((unsigned)((C + 31) / 32), (unsigned)((R + TR - 1) / TR));
  const uint8_t* from = static_cast<const uint8_t*>(in);
  uint8_t* to = static_cast<uint8_t*>(out);
  if (((uintptr_t)in & 3u) == 0 && in_ld * S % 4 == 0)
    pe_transpose_kernel<S, true><<<grid, 128, 0, stream>>>(from, to, R, C, in_ld, out_ld);
  else
    pe_transpose_kernel<S, S == 4><<<grid, 128, 0, stream>>>(from, to, R, C, in_ld, out_ld);
}

}  // namespace

int launch_team(const pe_graph* g, const Plan& p, bool by_pos, int64_t K, const uint8_t* assign, const uint16_t* order,
                uint32_t flags, const pe_outputs& out, void* workspace, cudaStream_t stream, int64_t* launches) {
  TeamCall t;
  t.g = g; t.p = &p; t.K = K; t.flags = flags; t.stream = stream;
  if (!p.staged) {
    t.kc = K; t.assign = assign; t.order = order; t.out = out;
    t.sd.in_row = (size_t)K; t.sd.in_cand = 1; t.sd.out_row = (size_t)K; t.sd.out_cand = 1;
    *launches += 1;
    return by_pos ? launch1<true>(t) : launch1<false>(t);
  }
  // staged: chunks of candidates go through candidate-major copies in the workspace, which has room for two
  // chunks.  Evaluations alternate between two streams, so that the tail of one overlaps the head of the next; the
  // transpositions have a stream of higher priority of their own: their blocks are placed in what the evaluation's
  // blocks leave free of an SM (at the same priority they wait until every block of an evaluation is placed).
  const int64_t V = g->V, Vp = p.team_vp;
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  const bool times = out.start != nullptr;
  const bool fork = K > p.team_chunk;
  pe_graph* gm = const_cast<pe_graph*>(g);
  std::unique_lock<std::mutex> lock(gm->team_mutex, std::defer_lock);
  bool ok = true;
  auto record = [&](cudaEvent_t e, cudaStream_t s) { if (fork) ok = cudaEventRecord(e, s) == cudaSuccess && ok; };
  auto wait = [&](cudaStream_t s, cudaEvent_t e) { if (fork) ok = cudaStreamWaitEvent(s, e, 0) == cudaSuccess && ok; };
  const cudaStream_t copies = fork ? gm->team_copy : stream;
  if (fork) lock.lock();
  record(gm->team_fork, stream);
  wait(gm->team_stream[0], gm->team_fork);
  wait(gm->team_stream[1], gm->team_fork);
  wait(gm->team_copy, gm->team_fork);
  auto half_of = [&](int q) { return ws + (size_t)(q & 1) * p.team_half; };
  auto copy_back = [&](int q, int64_t c0) {   // times of chunk q, once it is evaluated
    const int64_t kc = K - c0 < p.team_chunk ? K - c0 : p.team_chunk;
    wait(copies, gm->team_done[q & 1]);
    transpose<4>(half_of(q) + p.team_off_start, out.start + c0, kc, V, Vp, K, copies);
    transpose<4>(half_of(q) + p.team_off_finish, out.finish + c0, kc, V, Vp, K, copies);
    record(gm->team_back[q & 1], copies);
    *launches += 2;
  };
  int rc = PE_OK;
  int q = 0;
  for (int64_t c0 = 0; c0 < K && rc == PE_OK; c0 += p.team_chunk, ++q) {
    const int64_t kc = K - c0 < p.team_chunk ? K - c0 : p.team_chunk;
    uint8_t* half = half_of(q);
    uint16_t* ord_t = reinterpret_cast<uint16_t*>(half + p.team_off_order);
    uint8_t* asg_t = half + p.team_off_assign;
    t.stream = fork ? gm->team_stream[q & 1] : stream;
    if (q >= 2) wait(copies, gm->team_done[q & 1]);     // chunk q - 2 has read its inputs
    transpose<2>(order + c0, ord_t, V, kc, K, Vp, copies);
    transpose<1>(assign + c0, asg_t, V, kc, K, Vp, copies);
    record(gm->team_in[q & 1], copies);
    wait(t.stream, gm->team_in[q & 1]);
    if (q >= 2 && times) wait(t.stream, gm->team_back[q & 1]);   // the times of chunk q - 2 have left
    t.kc = kc; t.assign = asg_t; t.order = ord_t;
    t.out.start = times ? reinterpret_cast<int32_t*>(half + p.team_off_start) : nullptr;
    t.out.finish = times ? reinterpret_cast<int32_t*>(half + p.team_off_finish) : nullptr;
    t.out.makespan = out.makespan ? out.makespan + c0 : nullptr;
    t.out.status = out.status ? out.status + c0 : nullptr;
    t.out.busy = out.busy ? out.busy + c0 : nullptr;
    t.out.peak_mem = out.peak_mem ? out.peak_mem + c0 : nullptr;
    t.sd.in_row = 1; t.sd.in_cand = (size_t)Vp; t.sd.out_row = 1; t.sd.out_cand = (size_t)Vp;
    rc = by_pos ? launch1<true>(t) : launch1<false>(t);
    record(gm->team_done[q & 1], t.stream);
    *launches += 3;
    if (rc == PE_OK && times && q >= 1) copy_back(q - 1, c0 - p.team_chunk);
  }
  if (rc == PE_OK && times) copy_back(q - 1, (int64_t)(q - 1) * p.team_chunk);
  // join, also after an error: nothing of this call may stay unordered on the side streams
  record(gm->team_join[0], gm->team_stream[0]);
  record(gm->team_join[1], gm->team_stream[1]);
  record(gm->team_join[2], gm->team_copy);
  for (int b = 0; b < 3; ++b) wait(stream, gm->team_join[b]);
  if (!ok && rc == PE_OK) rc = PE_ERR_CUDA;
  return rc;
}

}  // namespace pe
