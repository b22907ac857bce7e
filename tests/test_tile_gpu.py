"""The lane-per-candidate kernel at the edges of its tiles: batches around a tile of 32 (or fewer) candidates and one
that no four-candidate load divides, orders whose length leaves every kind of remainder of the request blocks, 16- and
32-bit state words, tiles narrower than a warp, each form of the link-class encoding, candidates that are invalid in
one lane only.  Integers: bit-exact against the oracle."""
import numpy as np
import pytest

from paper_2503_09357_b200 import workloads as wl
from tests import checkers as ck
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


def chain_graph(V, D, indeg, classes, scale, seed=0):
    rs = np.random.RandomState(seed + V)
    edges = [(int(p), i) for i in range(1, V) for p in rs.choice(i, size=min(i, indeg), replace=False)]
    cls = None if classes == 1 else rs.randint(0, 2, (D, D)).astype(np.uint8)
    if classes == 3:
        cls[0, D - 1] = 0xFF
    L = 1 if classes == 1 else 2
    w = ck.problem(V, edges, rs.randint(0, scale, V), D, comm=rs.randint(0, scale, (len(edges), L)) if edges else None,
                   L=L, link_class=cls, A=rs.randint(-4, 5, V), W=rs.randint(0, 3, V) if V % 2 else None,
                   cap=rs.randint(5, 60, D))
    w.assign_mode, w.group = "per_op", None
    return w


@pytest.mark.parametrize("V,D,indeg,classes,scale,K", [
    (15, 3, 2, 1, 4, 31), (16, 3, 2, 1, 4, 33), (17, 4, 3, 1, 4, 64), (47, 8, 3, 1, 200, 128), (48, 8, 2, 2, 200, 129),
    (49, 40, 3, 2, 30, 96), (63, 32, 5, 2, 30, 97), (65, 5, 6, 1, 300, 1), (80, 6, 3, 3, 30, 4740), (1500, 8, 3, 1, 40, 300),
    (1600, 8, 2, 2, 40, 299), (1200, 8, 6, 3, 9, 301), (1100, 12, 6, 1, 9, 200)])
def test_tile_edges_match_the_oracle(V, D, indeg, classes, scale, K):
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2503_09357_b200 import binding as pe
    w = chain_graph(V, D, indeg, classes, scale)
    assign, order = wl.make_candidates(w, K=K)
    if K > 40:                                          # one lane each: an operator twice in a row, a predecessor late,
        order[5, 3] = order[4, 3]                       # no operator, a machine that does not exist
        order[:, 6] = order[::-1, 6].copy()
        order[7, 9] = 65535
        assign[int(order[V // 2, 11]), 11] = 255
    g = pe.Graph(w)
    try:
        for flags in (0, pe.PE_ASSIGN_BY_POS | pe.PE_TIMES_BY_OP, pe.PE_COMM_EXCLUSIVE):
            a = assign
            if flags & pe.PE_ASSIGN_BY_POS:
                a = np.take_along_axis(assign, np.minimum(order, V - 1).astype(np.int64), axis=0)
            if pe.pe_eval_variant(g.handle, K, flags | pe.PE_VARIANT_SHARED) < 0:
                continue
            gu.check(g, w, a, order, flags=flags | pe.PE_VARIANT_SHARED, label=f"flags {flags}")
    finally:
        g.close()


@pytest.mark.parametrize("by_pos", [False, True])
@pytest.mark.parametrize("dur,scale", [(65535, 1), (255, 0)])
def test_repetitions_behind_a_missing_source_are_flagged(dur, scale, by_pos):
    """Operator 0 is placed again and again ahead of its predecessor: every repetition adds its duration to a time that
    is beyond all reachable ones, until the packed word wraps into the reachable range.  `repeat` covers the count (129)
    at which that happens, with 32-bit words (dur 65535) and, where the time bound allows, 16-bit words (dur 255)."""
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2503_09357_b200 import binding as pe
    V, D, K = 310, 2, 300
    w = ck.problem(V, [(1, 0)], np.where(np.arange(V) == 0, dur, scale), D, comm=0)
    w.assign_mode, w.group = "per_op", None
    assign = np.ones((V, K), np.uint8)
    assign[0] = 0
    order = np.repeat((2 + np.arange(V) % (V - 2)).astype(np.uint16)[:, None], K, axis=1)
    for c in range(K):
        repeat = 2 + c // 2
        if c % 2:
            order[V - repeat:, c] = 0                   # one after the other at the end,
        else:
            order[V - 2 * repeat + 1::2, c] = 0         # or with another operator in between
    a = np.take_along_axis(assign, order.astype(np.int64), axis=0) if by_pos else assign
    g = pe.Graph(w)
    try:
        gpu, ref = gu.check(g, w, a, order, flags=pe.PE_VARIANT_SHARED | (pe.PE_ASSIGN_BY_POS if by_pos else 0))
        assert (ref["status"] & pe.PE_STATUS_ORDER_INVALID).all()
    finally:
        g.close()


@pytest.mark.parametrize("top,classes,indeg", [(0x7FFFFE, 1, 3), (0x7FFFFF, 1, 3), (0xFFFEFF, 1, 2), (0xFFFEFF, 2, 5), (0xFFFEFF, 3, 3)])
def test_time_bounds_up_to_24_bits(top, classes, indeg):
    """Sum of durations and delays just below and at the bound from which a sum with the unscheduled word may wrap, and at
    the largest that fits a packed word: the lane kernel still serves them, with and without exclusive channels."""
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2503_09357_b200 import binding as pe
    V, D, K = 300, 5, 130
    w = chain_graph(V, D, indeg, classes, 2, seed=top % 97)
    w.comm[:] = w.comm * 3000
    rest = top - int(w.comm.max(axis=1).sum())
    w.dur = np.full(V, rest // V, np.int32)
    w.dur[V - 1] += rest - int(w.dur.sum())
    assert w.dur.max() <= 65535 and int(w.dur.sum()) + int(w.comm.max(axis=1).sum()) == top
    assign, order = wl.make_candidates(w, K=K)
    order[5, 3] = order[4, 3]
    order[:, 6] = order[::-1, 6].copy()
    order[7, 9] = 65535
    order[-140:, 12] = order[-141, 12]
    g = pe.Graph(w)
    try:
        for flags in (0, pe.PE_ASSIGN_BY_POS, pe.PE_COMM_EXCLUSIVE, pe.PE_ASSIGN_BY_POS | pe.PE_COMM_EXCLUSIVE):
            a = assign
            if flags & pe.PE_ASSIGN_BY_POS:
                a = np.take_along_axis(assign, np.minimum(order, V - 1).astype(np.int64), axis=0)
            gu.check(g, w, a, order, flags=flags | pe.PE_VARIANT_SHARED, label=f"flags {flags}")
            gu.check(g, w, a, order, flags=flags | pe.PE_VARIANT_SHARED | pe.PE_TIMES_BY_OP, label=f"flags {flags} by op")
            gu.check(g, w, a, order, flags=flags, label=f"auto {flags}")
    finally:
        g.close()


def test_more_candidates_than_2_to_the_26():
    """Row pitches in bytes near the top of 32 bits' halves; two operators, so that the result can be written down."""
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2503_09357_b200 import binding as pe
    K = (1 << 26) + 37
    w = ck.problem(2, [], [3, 5], 2)
    g = pe.Graph(w)
    try:
        gen = torch.Generator(device="cuda"); gen.manual_seed(1)
        assign = torch.randint(0, 2, (2, K), dtype=torch.uint8, device="cuda", generator=gen)
        order = torch.randint(0, 2, (1, K), dtype=torch.int16, device="cuda", generator=gen)
        order = torch.cat([order, 1 - order])
        for flags in (pe.PE_VARIANT_SHARED, pe.PE_VARIANT_SHARED | pe.PE_TIMES_BY_OP | pe.PE_COMM_EXCLUSIVE):
            out = g.eval_batch(assign, order, flags=flags)
            same = assign[0] == assign[1]
            assert int(out["status"].abs().max()) == 0
            assert torch.equal(out["makespan"], torch.where(same, 8, 5).to(torch.int32))
            first = order[0] if not flags & pe.PE_TIMES_BY_OP else torch.zeros_like(order[0])
            ahead = same & (order[0] != first)
            want = torch.where(first == 0, 3, 5).to(torch.int32) + torch.where(ahead, torch.where(first == 0, 5, 3), 0).to(torch.int32)
            assert torch.equal(out["finish"][0], want)
    finally:
        g.close()


@pytest.mark.parametrize("V,D,indeg,classes,scale,K,hetero", [
    (48, 8, 2, 2, 4, 129, False), (49, 40, 3, 2, 30, 96, False), (256, 8, 3, 1, 4, 4741, False), (1500, 8, 3, 1, 40, 301, False),
    (65, 5, 6, 1, 300, 33, True), (80, 6, 3, 3, 30, 300, True), (700, 12, 2, 2, 30, 201, True)])
def test_every_form_runs_on_the_lane_kernel(V, D, indeg, classes, scale, K, hetero):
    """Every layout of assignments and times on the lane kernel itself: the shared variant needs no workspace and, unlike
    the generic kernel behind the same name, serves batches whose times are both wanted or both absent."""
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2503_09357_b200 import binding as pe
    w = chain_graph(V, D, indeg, classes, scale, seed=7)
    if hetero:
        w.dur_by_machine = np.random.RandomState(V).randint(0, scale, (V, D)).astype(np.int32)
    assign, order = wl.make_candidates(w, K=K)
    order[5, 3] = order[4, 3]
    order[7, 9] = 65535
    assign[int(order[V // 2, 11]), 11] = 255
    a_pos = np.take_along_axis(assign, np.minimum(order, V - 1).astype(np.int64), axis=0)
    g = pe.Graph(w)
    try:
        base = (0, pe.PE_TIMES_BY_OP, pe.PE_ASSIGN_BY_POS, pe.PE_ASSIGN_BY_POS | pe.PE_TIMES_BY_OP)
        exclusive = () if hetero or D > 32 or V > 1000 else tuple(f | pe.PE_COMM_EXCLUSIVE for f in base)
        for flags in base + exclusive:
            assert pe.pe_eval_variant(g.handle, K, flags | pe.PE_VARIANT_SHARED) == pe.PE_VARIANT_SHARED
            for want_times in (True, False):
                gu.check(g, w, a_pos if flags & pe.PE_ASSIGN_BY_POS else assign, order, flags=flags | pe.PE_VARIANT_SHARED,
                         want_times=want_times, label=f"flags {flags} times {want_times}")
    finally:
        g.close()
