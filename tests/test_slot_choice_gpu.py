"""Where the automatic choice takes the slot kernels, and what it asks for them."""
import numpy as np
import pytest

from paper_2503_09357_b200 import workloads as wl
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


def binding():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2503_09357_b200 import binding as pe
    return pe


def launches(pe, g, w, K, flags=0, want_times=True, workspace=None):
    """Kernels that one call launches, checked against the oracle."""
    assign, order = wl.make_candidates(w, K=K)
    if flags & pe.PE_ASSIGN_BY_POS:
        assign = np.take_along_axis(assign, order.astype(np.int64), axis=0)
    if workspace is None:
        before = pe.pe_kernel_launches()
        gu.check(g, w, assign, order, flags=flags, want_times=want_times)
        return pe.pe_kernel_launches() - before
    import torch
    from oracle import pe_oracle as orc
    out = g.alloc_outputs(K, want_times)
    before = pe.pe_kernel_launches()
    g.eval_batch(torch.from_numpy(assign).cuda(), torch.from_numpy(gu.as_signed(order)).cuda(), flags=flags, out=out, workspace=workspace)
    torch.cuda.synchronize()
    n = pe.pe_kernel_launches() - before
    res = {k: v.cpu().numpy() for k, v in out.items()}
    res["status"] = res["status"].view(np.uint32)
    gu.compare(res, orc.evaluate(w, assign, order, flags=flags & 7, want_times=want_times, threads=gu.CPU_THREADS))
    return n


@pytest.mark.parametrize("config,kw,K", [(1, {}, 1024), (5, dict(V=256, D=8), 1 << 20), (1, {}, 65536)])
def test_batches_that_never_take_the_slot_kernels_ask_for_nothing(config, kw, K):
    """(Half a batch of the bidirectional pipeline at K = 65536 may take them: K = 32768 without times.)"""
    pe = binding()
    g = pe.Graph(wl.make_config(config, **kw))
    try:
        assert pe.pe_workspace_bytes(g.handle, K, 0) == 0
        assert pe.pe_workspace_bytes(g.handle, K, 1 << 20) == 0   # (flags that no call accepts)
    finally:
        g.close()


def test_workspace_is_what_the_slot_kernels_use():
    """Multi-modal graph: 4 bytes a position and a status word, a candidate."""
    pe = binding()
    w = wl.make_config(4)
    V, K = w.num_ops, 8192
    g = pe.Graph(w)
    try:
        per = V * 4 + 4 + (w.num_devices * 4 if w.mem_weight is not None else 0)
        import torch
        n = pe.pe_workspace_bytes(g.handle, K, 0)
        assert K * per <= n <= K * per + 4096
        ws = torch.empty(n, dtype=torch.uint8, device="cuda")
        # the workspace of the largest batch serves the smaller ones, whichever kernel they take
        for k, want in ((K, 2), (4097, None), (1001, None), (64, None), (1, None)):
            got = launches(pe, g, w, k, workspace=(ws, n))
            assert want is None or got == want
    finally:
        g.close()


@pytest.mark.parametrize("K,kernels", [(148, 1), (1000, 1), (9472, 2)])
def test_small_batches_of_operators_with_many_sources_take_a_warp_each(K, kernels):
    """Sixteen sources an operator: a lane walks them one after the other (955 us at any small K), a warp side by side (522)."""
    pe = binding()
    w = wl.make_config(3, layers=16, experts=16, microbatches=4)
    g = pe.Graph(w)
    try:
        assert launches(pe, g, w, K) == kernels
    finally:
        g.close()


@pytest.mark.parametrize("K", [148, 4096])
def test_exclusive_channels_of_the_tiny_pipeline_stay_with_the_lane_kernel(K):
    """One launch (20 us) instead of two (24 us)."""
    pe = binding()
    w = wl.make_config(1)
    g = pe.Graph(w)
    try:
        for times in (True, False):
            assert launches(pe, g, w, K, pe.PE_COMM_EXCLUSIVE, times) == 1
    finally:
        g.close()


@pytest.mark.parametrize("V,D,by_pos,kernels", [(484, 64, False, 2), (529, 64, False, 1), (1024, 64, True, 2)])
def test_larger_graphs_with_marks_need_no_workspace_by_operator(V, D, by_pos, kernels):
    pe = binding()
    w = wl.make_config(5, V=V, D=D)
    flags = pe.PE_ASSIGN_BY_POS if by_pos else 0
    g = pe.Graph(w)
    try:
        assert launches(pe, g, w, 16384, flags) == kernels
        assert (pe.pe_workspace_bytes(g.handle, 16384, flags) == 0) == (kernels == 1)
    finally:
        g.close()


def test_an_unaligned_workspace_is_left_alone():
    """The slot kernels use 16-byte accesses; other kernels run where the workspace does not allow for those."""
    import torch
    pe = binding()
    w = wl.make_config(4, microbatches=4)
    K = 16384
    g = pe.Graph(w)
    try:
        n = pe.pe_workspace_bytes(g.handle, K, 0)
        ws = torch.empty(n + 256, dtype=torch.uint8, device="cuda")
        assert launches(pe, g, w, K, workspace=(ws, n)) == 2
        assert launches(pe, g, w, K, workspace=(ws[8:], n)) == 1
    finally:
        g.close()


@pytest.mark.parametrize("config,kw,K,flag,kernel,n", [
    (4, {}, 8192, None, "pe_eval_slot_kernel", 2), (3, {}, 8192, "PE_TIMES_BY_OP", "pe_eval_slot_kernel", 3),
    (4, {}, 8192, "PE_VARIANT_SHARED", "pe_eval_tile_kernel", 1), (4, {}, 64, None, "pe_eval_team_kernel", 1),
    (4, {}, 64, "PE_VARIANT_WARP", "pe_eval_warp2_kernel", 1), (4, {}, 64, "PE_VARIANT_GLOBAL", "pe_eval_lane_kernel", 1)])
def test_the_kernel_that_is_named_is_the_one_that_runs(config, kw, K, flag, kernel, n):
    pe = binding()
    w = wl.make_config(config, **kw)
    g = pe.Graph(w)
    try:
        flags = getattr(pe, flag) if flag else 0
        assert pe.pe_eval_kernel(g.handle, K, flags) == kernel
        assert launches(pe, g, w, K, flags) == n
        assert pe.pe_eval_kernel(g.handle, K, 1 << 20) is None
    finally:
        g.close()
