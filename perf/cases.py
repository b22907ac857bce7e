"""What is measured: calls that a user of the plan evaluator makes, over the range of graphs, batch sizes and options
that the package serves.

A case names an operator graph of `paper_2503_09357_b200.workloads` (with its own sizes), the number of candidate plans
K, the call and its options.  Calls:
  eval     pe_eval_batch over a resident batch with outputs and workspace that the program keeps;
  search   one generation of a search over priority lists as `search.py` runs it: decode the lists, evaluate without
           times, pick the elite and the best;
  host     pe_eval_batch_host: inputs from and outputs to pinned host memory.
Options: times (start and finish wanted, or the summary outputs only), by_pos (machine ids by position), times_by_op,
exclusive (one transfer per channel at a time), hetero (durations that depend on the machine).

Candidates have the distribution of `workloads/candgen.cpp`: a random key per operator, the ready operator with the
smallest key first; machines uniform per operator, or a random permutation of the pipeline slots.
"""
import random

import torch

from paper_2503_09357_b200 import binding as pe
from paper_2503_09357_b200 import workloads as wl


def _case(name, graph, K, call="eval", times=True, by_pos=False, times_by_op=False, exclusive=False, hetero=False, **size):
    return dict(name=name, graph=graph, K=K, call=call, times=times, by_pos=by_pos, times_by_op=times_by_op,
                exclusive=exclusive, hetero=hetero, **size)


def listed():
    return [
        # the smallest call: one batch of the tiny pipeline (latency and launches)
        _case("eval_tiny_K1024", "tiny", 1024, S=4, M=8),
        # a generation of a search over a small pipeline: many short calls one after the other
        _case("search_tiny_K1024", "tiny", 1024, call="search", times=False, S=4, M=8),
        # a generation of a search over a real model graph (vision and text encoders, decoder)
        _case("search_multimodal_K8192", "multimodal", 8192, call="search", times=False, microbatches=8),
        # the bidirectional pipeline schedule, a full batch
        _case("eval_bidirectional_K65536", "bidirectional", 65536, P=8, M=20),
        # the same graph on machines of different speed
        _case("eval_bidirectional_hetero_K16384", "bidirectional", 16384, hetero=True, P=8, M=20),
        # many candidates of a small random graph
        _case("eval_V256_D8_K1M", "layered", 1 << 20, side=16, D=8),
        # a middle-sized graph on many machines, assignments as machine sequences
        _case("eval_V1024_D64_bypos_K512k", "layered", 1 << 19, by_pos=True, side=32, D=64),
        # the multi-modal model, a full batch with start and finish of every operator
        _case("eval_multimodal_K65536", "multimodal", 65536, microbatches=8),
        # the same model when channels carry one transfer at a time, only the figures that a search ranks by
        _case("eval_multimodal_exclusive_K16384", "multimodal", 16384, times=False, exclusive=True, microbatches=8),
        # mixture of experts (operators with eight inputs), an odd batch, times by operator
        _case("eval_moe_K16381", "moe", 16381, times_by_op=True, layers=32, experts=8, microbatches=4),
        # from and to host memory
        _case("host_moe_K16384", "moe", 16384, call="host", layers=32, experts=8, microbatches=4),
        # the largest graph, a full batch
        _case("eval_V16384_D64_K65536", "layered", 65536, side=128, D=64),
    ]


def draw(rng: random.Random):
    """One more case: a graph of any of the five families, a call, options, and a batch size spread over its logarithm."""
    graph = rng.choice(["tiny", "bidirectional", "multimodal", "moe", "layered", "layered"])
    if graph == "tiny":
        size = dict(S=rng.randint(2, 8), M=rng.randint(2, 16))
        V = 2 * size["S"] * size["M"]
    elif graph == "bidirectional":
        size = dict(P=2 * rng.randint(1, 8), M=2 * rng.randint(1, 20))
        V = 3 * size["P"] * size["M"]
    elif graph == "multimodal":
        size = dict(microbatches=rng.randint(1, 12))
        V = 192 * size["microbatches"]
    elif graph == "moe":
        size = dict(layers=rng.randint(4, 32), experts=rng.choice([4, 8]), microbatches=rng.randint(1, 4))
        V = 2 * size["layers"] * (size["experts"] + 3) * size["microbatches"]
    else:
        size = dict(side=int(round(16 * 8 ** rng.random())), D=rng.choice([4, 8, 16, 32, 64]))
        V = size["side"] ** 2
    call = rng.choice(["eval", "eval", "eval", "eval", "search", "host"])
    hetero = exclusive = False
    if call != "host":
        option = rng.random()
        exclusive = option < 0.1
        hetero = 0.1 <= option < 0.2
    log_most = 28.0 if call == "eval" and not (hetero or exclusive) else 25.0      # log2 of V * K
    ops = 2.0 ** rng.uniform(16.0, log_most)
    K = max(1, int(ops / V))
    if rng.random() < 0.5:
        K = max(4, K // 4 * 4)
    return dict(graph=graph, K=K, call=call, times=call != "search" and rng.random() < 0.7, by_pos=call != "search" and rng.random() < 0.25,
                times_by_op=call != "search" and rng.random() < 0.25, exclusive=exclusive, hetero=hetero, **size)


def _workload(case):
    kind = case["graph"]
    if kind == "tiny":
        w = wl.make_config(1, S=case["S"], M=case["M"])
    elif kind == "bidirectional":
        w = wl.make_config(2, P=case["P"], M=case["M"])
    elif kind == "moe":
        w = wl.make_config(3, layers=case["layers"], experts=case["experts"], microbatches=case["microbatches"])
    elif kind == "multimodal":
        w = wl.make_config(4, microbatches=case["microbatches"])
    else:
        w = wl.make_config(5, V=case["side"] ** 2, D=case["D"])
    if case["hetero"]:
        # machine j runs an operator in 1, 1.25, 1.5 or 1.75 times its duration
        import numpy as np
        slow = 4 + np.arange(w.num_devices) % 4
        w.dur_by_machine = np.ascontiguousarray((w.dur[:, None].astype(np.int64) * slow[None, :] // 4).astype(np.int32))
    return w


def _flags(case):
    return ((pe.PE_ASSIGN_BY_POS if case["by_pos"] else 0) | (pe.PE_TIMES_BY_OP if case["times_by_op"] else 0) |
            (pe.PE_COMM_EXCLUSIVE if case["exclusive"] else 0))


def _lists(w, K, gen):
    """Uniformly random priority lists, int16 bits [V, K]."""
    V = w.num_ops
    out = torch.empty((V, K), dtype=torch.int16, device="cuda")
    step = max(1, (1 << 26) // V)
    for c in range(0, K, step):
        n = min(step, K - c)
        out[:, c:c + n] = torch.rand((n, V), device="cuda", generator=gen).argsort(dim=1).to(torch.int16).t()
    return out


def _assign(w, K, gen):
    D = w.num_devices
    if w.assign_mode == "group_perm":
        perm = torch.rand((D, K), device="cuda", generator=gen).argsort(dim=0).to(torch.uint8)
        return perm[torch.from_numpy(w.group).cuda().long()].contiguous()
    return torch.randint(0, D, (w.num_ops, K), dtype=torch.uint8, device="cuda", generator=gen)


def _order(graph, lists):
    """The topological orders of the lists, a slice of candidates at a time (bounded workspace)."""
    V, K = lists.shape
    step = max(4, (1 << 28) // V)
    if K <= step:
        return graph.decode_priority(lists)[0]
    out = torch.empty_like(lists)
    for c in range(0, K, step):
        out[:, c:c + step] = graph.decode_priority(lists[:, c:c + step].contiguous())[0]
    return out


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    w = _workload(case)
    K = case["K"]
    graph = pe.Graph(w)
    flags = _flags(case)
    lists = _lists(w, K, gen)
    assign = _assign(w, K, gen)
    st = dict(call=case["call"], graph=graph, K=K, flags=flags, elite=max(1, K // 8))
    if case["call"] == "search":
        st.update(lists=lists, assign=assign)
        return st
    order = _order(graph, lists)
    del lists
    if case["by_pos"]:
        step = max(1, (1 << 26) // w.num_ops)
        for c in range(0, K, step):
            assign[:, c:c + step] = assign[:, c:c + step].gather(0, order[:, c:c + step].long() & 0xFFFF)
    st.update(out=graph.alloc_outputs(K, case["times"]), workspace=graph.alloc_workspace(K, flags))
    if case["call"] == "host":
        st.update(host_assign=assign.cpu().pin_memory(), host_order=order.cpu().pin_memory(),
                  host_out={k: torch.empty(v.shape, dtype=v.dtype).pin_memory() for k, v in st["out"].items()})
    st.update(assign=assign, order=order)
    return st


def run(st):
    g = st["graph"]
    if st["call"] == "eval":
        return g.eval_batch(st["assign"], st["order"], flags=st["flags"], out=st["out"], workspace=st["workspace"])
    if st["call"] == "search":
        order, list_status = g.decode_priority(st["lists"])
        out = g.eval_batch(st["assign"], order, flags=st["flags"], want_times=False)
        out["status"] |= list_status
        elite, count = g.select_topk(out, st["elite"])
        best, makespan, qualifying = g.select_best(out)
        return dict(out, order=order, elite=elite, count=count, best=best, best_makespan=makespan, qualifying=qualifying)
    host, dev = (pe.make_outputs(**{k: v.data_ptr() for k, v in st[name].items()}) for name in ("host_out", "out"))
    ws, ws_bytes = st["workspace"]
    rc = pe.pe_eval_batch_host(g.handle, st["K"], st["host_assign"].data_ptr(), st["host_order"].data_ptr(), 2, st["flags"],
                               host, st["assign"].data_ptr(), st["order"].data_ptr(), dev, ws.data_ptr(), ws_bytes,
                               torch.cuda.current_stream().cuda_stream)
    if rc != pe.PE_OK:
        raise pe.PeError(rc, "pe_eval_batch_host")
    return st["host_out"]


def work(case):
    w = _workload(case)
    V, E, D, K = w.num_ops, w.num_edges, w.num_devices, case["K"]
    # machine id (1) and order entry (2) in, start and finish (4 + 4) out; makespan, status, busy[D], peak[D] per candidate
    per_op = 3 + (8 if case["times"] else 0)
    if case["call"] == "search":
        per_op += 2                      # the list comes in, the order goes out
    nbytes = K * V * per_op + K * (8 + 8 * D)
    return {"bytes": float(nbytes), "flops": float(K) * (2.0 * E + 6.0 * V)}


def tolerance(case):
    return "exact"                       # int32 throughout; every output is determined
