"""The lane-per-candidate decoder at the edges of its range: 8-bit ids (V = 255, 256), bitmap words, blocks of 128
candidates, an operator with 255 predecessors, lists that are no permutation.  Bit-exact against the oracle."""
import numpy as np
import pytest

from paper_2503_09357_b200 import workloads as wl
from tests import checkers as ck
from tests import gpu_util as gu
from tests.test_decode_gpu import gpu_decode, random_lists

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,fan,K", [(1, 0, 129), (31, 2, 20001), (33, 3, 20000), (64, 2, 16384), (255, 3, 20001),
                                     (256, 255, 20033), (256, 2, 16385), (257, 2, 16385)])
def test_small_graphs_in_large_batches(V, fan, K):
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from oracle import pe_oracle as orc
    from paper_2503_09357_b200 import binding as pe
    rs = np.random.RandomState(V + fan)
    if fan == 255:
        edges = [(i, V - 1) for i in range(V - 1)]
    else:
        edges = [(int(p), i) for i in range(1, V) for p in rs.randint(0, i, size=min(i, fan))]   # duplicates allowed
    w = ck.problem(V, edges, rs.randint(1, 9, V), 2)
    w.assign_mode, w.group = "per_op", None
    plist = random_lists(V, K, V)
    if V > 2:
        plist[1, 5] = plist[0, 5]
        plist[2, K - 1] = V
    ref_order, ref_status = orc.decode(w, plist, threads=gu.CPU_THREADS)
    g = pe.Graph(w)
    try:
        order, status = gpu_decode(g, plist)
        assert np.array_equal(status, ref_status)
        ok = ref_status == 0
        assert np.array_equal(order[:, ok], ref_order[:, ok])
    finally:
        g.close()
