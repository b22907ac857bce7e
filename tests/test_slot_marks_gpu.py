"""The slot kernels on graphs with many operators that nobody follows: such an operator leaves a mark in a predecessor's
state word, and every operator checks the word of its own slot.  One to three sources an operator, machine ids by operator
and by position, times by position, by operator and none, durations by machine, odd batches, weights, and candidates that are
invalid in one lane only.  Every call has to go through the slot kernels.  Integers: bit-exact against the oracle."""
import numpy as np
import pytest

from paper_2503_09357_b200 import workloads as wl
from tests import checkers as ck
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


def leafy_graph(V, fan, D, scale):
    """Every second operator has no successors: without marks more than a quarter of the operators would need a word of
    their own.  Operator ids are shuffled.  Returns the problem and the ids in a topological order."""
    rs = np.random.RandomState(V * 10 + fan)
    ids = rs.permutation(V)
    width = 6
    edges = []
    for i in range(V):
        core = i // 2                      # operators 2c are the core, 2c + 1 the leaves
        last = core - width if i % 2 == 0 else core
        if last < 0:
            continue
        first = max(0, last - 7)
        n = fan if i > V // 2 and i < V // 2 + 4 else rs.randint(1, fan + 1)
        for c in {last} | set(int(x) for x in rs.choice(np.arange(first, last + 1), min(n - 1, last + 1 - first), replace=False)):
            edges.append((int(ids[2 * c]), int(ids[i])))
    indeg = np.bincount([e[1] for e in edges], minlength=V).max()
    assert indeg == fan
    w = ck.problem(V, edges, rs.randint(0, scale, V), D, comm=rs.randint(0, scale, (len(edges), 1)), A=rs.randint(-4, 5, V),
                   W=rs.randint(0, 3, V) if V % 2 else None, cap=rs.randint(5, 60, D))
    w.assign_mode, w.group = "per_op", None
    return w, ids


def spoil(w, assign, order, first):
    """Candidates from `first` on become invalid, each in its own way (some may stay valid: the oracle says)."""
    V, src, dst = w.num_ops, np.asarray(w.edge_src), np.asarray(w.edge_dst)
    rs = np.random.RandomState(V)
    follows = np.zeros(V, bool)
    follows[src] = True                                    # has successors

    def at(c, i):
        return int(np.flatnonzero(order[:, c] == i)[0])

    leaf = next(int(i) for i in dst if not follows[i])
    holder = int(src[dst == leaf][0])
    child = next(int(d) for s, d in zip(src, dst) if s == holder and follows[d])
    grandchild = next((int(d) for s, d in zip(src, dst) if s == child and follows[d]), child)
    other = next(int(i) for i in dst if not follows[i] and i != leaf)
    c = iter(range(first, order.shape[1]))
    q = next(c); order[at(q, other), q] = leaf                                                # a leaf twice, another one missing
    q = next(c); p = at(q, leaf); order[p, q], order[min(p + 1, V - 1), q] = leaf, leaf       # twice in a row
    q = next(c); a, b = at(q, leaf), at(q, holder); order[[a, b], q] = order[[b, a], q]       # before its predecessor
    q = next(c); order[at(q, child), q] = holder                                              # the holder of a slot twice
    q = next(c); order[at(q, leaf), q] = holder                                               # and in a leaf's place
    q = next(c); a, b = at(q, grandchild), at(q, holder); order[[a, b], q] = order[[b, a], q]   # the next holders early
    q = next(c); a, b = at(q, grandchild), at(q, child); order[[a, b], q] = order[[b, a], q]
    q = next(c); order[at(q, holder), q] = child                                              # a later holder instead of one
    q = next(c); order[at(q, leaf), q] = V                                                    # no operator
    q = next(c); order[at(q, holder), q] = 65535
    q = next(c); order[V - 1, q] = V
    q = next(c); order[0, q] = V
    q = next(c); order[:, q] = order[::-1, q].copy()
    q = next(c); order[V - 1, q] = order[0, q]
    q = next(c); order[:, q] = leaf
    q = next(c); order[:, q] = holder
    q = next(c); assign[leaf, q] = w.num_devices                                              # machines that do not exist
    q = next(c); assign[holder, q] = 255
    q = next(c); assign[leaf, q] = 255; order[at(q, leaf), q] = holder
    for _ in range(100):                                                                      # one random slip each
        q = next(c)
        a, b = rs.randint(0, V, 2)
        if rs.rand() < 0.5:
            order[[a, b], q] = order[[b, a], q]
        else:
            order[a, q] = order[b, q]
    return next(c)


@pytest.mark.parametrize("V,fan,D,K,hetero", [
    (500, 1, 64, 12000, False), (503, 1, 250, 20003, False), (503, 2, 128, 9002, False), (507, 2, 250, 28001, False),
    (511, 3, 64, 12000, False), (507, 3, 250, 28001, False), (401, 1, 8, 20000, True), (403, 2, 60, 12001, True),
    (406, 3, 60, 12002, True)])
def test_every_form_matches_the_oracle(V, fan, D, K, hetero):
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2503_09357_b200 import binding as pe
    w, _ = leafy_graph(V, fan, D, 40)
    if hetero:
        w.dur_by_machine = np.random.RandomState(V).randint(0, 40, (V, D)).astype(np.int32)
    assign, order = wl.make_candidates(w, K=K)
    spoil(w, assign, order, 5)
    order[V - 1, K - 1] = order[V - 2, K - 1]
    a_pos = np.take_along_axis(assign, np.minimum(order, V - 1).astype(np.int64), axis=0)
    g = pe.Graph(w)
    try:
        for flags in (0, pe.PE_TIMES_BY_OP, pe.PE_ASSIGN_BY_POS, pe.PE_ASSIGN_BY_POS | pe.PE_TIMES_BY_OP):
            for times in (True, False):
                before = pe.pe_kernel_launches()
                _, ref = gu.check(g, w, a_pos if flags & pe.PE_ASSIGN_BY_POS else assign, order, flags=flags, want_times=times,
                                  label=f"flags {flags} times {times}")
                # the gather and the recurrence, and the kernel that turns times by operator around
                assert pe.pe_kernel_launches() - before == 2 + bool(times and flags & pe.PE_TIMES_BY_OP), (flags, times)
        assert 60 < int(((ref["status"] & gu.INVALID) != 0).sum()) < 130
    finally:
        g.close()
