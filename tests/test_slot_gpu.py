"""The slot kernels (operators share state words; a gather kernel in front of the recurrence): every form of the link
classes, one source up to more than eight, orders whose length leaves every remainder of the request blocks, batches that
are and are not a multiple of four, weights, durations by machine, exclusive channels in 16 and 32 bits, and candidates
that are invalid in one lane only.  Integers: bit-exact against the oracle."""
import numpy as np
import pytest

from paper_2503_09357_b200 import workloads as wl
from tests import checkers as ck
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


def narrow_graph(V, width, fan, classes, D, scale, seed=0):
    """Operator i follows some of the `fan` operators that end `width` places before it: about width results are alive."""
    rs = np.random.RandomState(seed + V)
    edges = []
    for i in range(width, V):
        last = i - width
        for p in {last} | set(int(x) for x in rs.randint(max(0, last - fan + 1), last + 1, rs.randint(0, fan))):
            edges.append((p, i))
    cls = None if classes == 1 else rs.randint(0, 2, (D, D)).astype(np.uint8)
    if classes == 3:
        cls[0, D - 1] = 0xFF
    L = 1 if classes == 1 else 2
    w = ck.problem(V, edges, rs.randint(0, scale, V), D, comm=rs.randint(0, scale, (len(edges), L)), L=L, link_class=cls,
                   A=rs.randint(-4, 5, V), W=rs.randint(0, 3, V) if V % 2 else None, cap=rs.randint(5, 60, D))
    w.assign_mode, w.group = "per_op", None
    return w


def check_all(pe, w, K, forms, exclusive):
    """Every form against the oracle; returns how many of them went through the slot kernels (two launches or three)."""
    V = w.num_ops
    assign, order = wl.make_candidates(w, K=K)
    order[5, 3] = order[4, 3]                           # an operator twice in a row, a predecessor late, no operator, a
    order[:, 6] = order[::-1, 6].copy()                 # machine that does not exist, both, an operator twice far apart
    order[7, 9] = 65535
    assign[int(order[V // 2, 11]), 11] = 255
    order[V - 1, 12] = V
    assign[int(order[2, 12]), 12] = w.num_devices
    order[V - 1, K - 1] = order[0, K - 1]
    a_pos = np.take_along_axis(assign, np.minimum(order, V - 1).astype(np.int64), axis=0)
    g = pe.Graph(w)
    through = 0
    try:
        for flags in forms:
            for base in (flags, flags | pe.PE_COMM_EXCLUSIVE) if exclusive else (flags,):
                for want_times in (True, False):
                    before = pe.pe_kernel_launches()
                    gu.check(g, w, a_pos if base & pe.PE_ASSIGN_BY_POS else assign, order, flags=base, want_times=want_times,
                             label=f"flags {base} times {want_times}")
                    through += pe.pe_kernel_launches() - before == 2 + bool(want_times and base & pe.PE_TIMES_BY_OP)
    finally:
        g.close()
    return through


@pytest.mark.parametrize("V,width,fan,classes,D,scale,K,hetero", [
    (400, 8, 1, 1, 4, 40, 40000, False), (401, 12, 2, 1, 16, 9, 40001, False), (402, 9, 2, 1, 130, 9, 24002, False),
    (403, 12, 6, 1, 8, 9, 70003, False), (404, 10, 14, 1, 7, 9, 90004, False), (805, 16, 1, 2, 32, 40, 40004, False),
    (406, 8, 7, 2, 16, 20, 70006, False), (407, 10, 12, 2, 5, 9, 90000, False), (408, 12, 3, 3, 6, 30, 70000, False),
    (409, 10, 2, 1, 9, 30, 20001, True), (410, 10, 5, 2, 8, 30, 60004, True), (411, 10, 11, 3, 8, 30, 70003, True)])
def test_every_form_matches_the_oracle(V, width, fan, classes, D, scale, K, hetero):
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2503_09357_b200 import binding as pe
    w = narrow_graph(V, width, fan, classes, D, scale)
    if hetero:
        w.dur_by_machine = np.random.RandomState(V).randint(0, scale, (V, D)).astype(np.int32)
    forms = (0, pe.PE_TIMES_BY_OP, pe.PE_ASSIGN_BY_POS, pe.PE_ASSIGN_BY_POS | pe.PE_TIMES_BY_OP)
    through = check_all(pe, w, K, forms, exclusive=not hetero and D <= 32)
    assert through >= 4, through


@pytest.mark.parametrize("scale,K", [(60, 9001), (400, 9000)])
def test_exclusive_channels_with_short_and_long_words(scale, K):
    """Time bounds on both sides of 2^16: channel words of 16 and of 32 bits."""
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2503_09357_b200 import binding as pe
    w = narrow_graph(700, 12, 1, 2, 16, scale)
    bound = int(np.asarray(w.dur, np.int64).sum() + np.asarray(w.comm).max(axis=1).sum())
    assert (bound < 65536) == (scale == 60)
    assert check_all(pe, w, K, (pe.PE_COMM_EXCLUSIVE, pe.PE_COMM_EXCLUSIVE | pe.PE_ASSIGN_BY_POS), exclusive=False) == 4


def test_chains_longer_than_the_versions_and_batches_without_workspace():
    """One slot would hold 600 operators, more than a version counts; without workspace the batch takes another kernel."""
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from oracle import pe_oracle as orc
    from paper_2503_09357_b200 import binding as pe
    V, K = 1200, 20000
    w = ck.problem(V, [(i - 2, i) for i in range(2, V)], np.full(V, 60), 3, comm=np.full((V - 2, 1), 3))
    w.assign_mode, w.group = "per_op", None
    assign, order = wl.make_candidates(w, K=K)
    g = pe.Graph(w)
    try:
        before = pe.pe_kernel_launches()
        _, ref = gu.check(g, w, assign, order, label="workspace")
        assert pe.pe_kernel_launches() - before == 2
        a = torch.from_numpy(assign).cuda(); o = torch.from_numpy(gu.as_signed(order)).cuda()
        out = g.alloc_outputs(K)
        outs = pe.make_outputs(**{k: v.data_ptr() for k, v in out.items()})
        before = pe.pe_kernel_launches()
        assert pe.pe_eval_batch(g.handle, K, a.data_ptr(), o.data_ptr(), 2, 0, outs, 0, 0, 0) == pe.PE_OK
        assert pe.pe_kernel_launches() - before == 1
        torch.cuda.synchronize()
        res = {k: v.cpu().numpy() for k, v in out.items()}
        res["status"] = res["status"].view(np.uint32)
        gu.compare(res, ref, "no workspace")
    finally:
        g.close()


def forked_chains(V, D, scale):
    """Chains side by side that fork every twenty operators; the branch ends after eight.  One source an operator, and the word
    that its slot held before where a branch begins."""
    rs = np.random.RandomState(V)
    edges, ends, i = [], [-1] * 6, 0
    while i < V:
        for c in range(6):
            for step in range(20):
                if i >= V:
                    break
                if ends[c] >= 0:
                    edges.append((ends[c], i))
                ends[c] = i
                i += 1
                if step == 10:
                    at = ends[c]
                    for _ in range(8):
                        if i < V:
                            edges.append((at, i))
                            at = i
                            i += 1
    w = ck.problem(V, edges, rs.randint(0, scale, V), D, comm=rs.randint(0, scale, (len(edges), 1)), A=rs.randint(-4, 5, V),
                   cap=rs.randint(5, 60, D))
    w.assign_mode, w.group = "per_op", None
    return w


@pytest.mark.parametrize("V,width,fan,classes,D,scale,K", [
    (1000, 12, 1, 1, 16, 30, 9000), (1000, 0, 0, 1, 24, 30, 9002), (1001, 12, 2, 1, 32, 30, 9001), (1003, 12, 6, 1, 8, 9, 9003),
    (1004, 10, 14, 1, 7, 9, 16004), (1005, 16, 1, 2, 32, 30, 8004), (1006, 8, 7, 2, 16, 20, 9006), (1007, 10, 12, 2, 5, 9, 16000),
    (1009, 12, 9, 3, 6, 30, 16009), (1300, 12, 1, 3, 20, 30, 5000)])
def test_every_call_goes_through_the_slot_kernels(V, width, fan, classes, D, scale, K):
    """Graphs that leave a lane per candidate few lanes: all sixteen forms (layouts, times, exclusive channels) of one, two,
    three, up to eight and more sources over one link class, two of them and a class table."""
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2503_09357_b200 import binding as pe
    w = narrow_graph(V, width, fan, classes, D, scale) if width else forked_chains(V, D, scale)
    forms = (0, pe.PE_TIMES_BY_OP, pe.PE_ASSIGN_BY_POS, pe.PE_ASSIGN_BY_POS | pe.PE_TIMES_BY_OP)
    assert check_all(pe, w, K, forms, exclusive=True) == 16
