"""Decoding with a pool of available operators, a lane per candidate: graphs that 1 to 32 chains cover, operators with many
successors and predecessors, the largest operator ids, odd batches, lists that are no permutation.  Bit-exact against the
oracle."""
import numpy as np
import pytest

from paper_2503_09357_b200 import workloads as wl
from tests import checkers as ck
from tests import gpu_util as gu
from tests.test_decode_gpu import gpu_decode, random_lists
from tests.test_slot_gpu import narrow_graph

pytestmark = pytest.mark.gpu


def check(w, K):
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from oracle import pe_oracle as orc
    from paper_2503_09357_b200 import binding as pe
    V = w.num_ops
    plist = random_lists(V, K, V)
    if K > 20 and V > 3:
        plist[1, 5] = plist[0, 5]
        plist[2, K - 1] = V
        plist[V - 1, 7] = 65535
    ref_order, ref_status = orc.decode(w, plist, threads=gu.CPU_THREADS)
    g = pe.Graph(w)
    try:
        order, status = gpu_decode(g, plist)
        assert np.array_equal(status, ref_status)
        ok = ref_status == 0
        assert np.array_equal(order[:, ok], ref_order[:, ok])
    finally:
        g.close()


@pytest.mark.parametrize("V,width,fan,K", [(3, 1, 1, 5), (300, 1, 1, 4097), (513, 7, 1, 4096), (700, 8, 3, 6001), (900, 16, 6, 4003),
                                           (777, 24, 14, 3000), (1000, 31, 2, 3001), (1024, 32, 20, 2049), (4095, 8, 2, 1500),
                                           (4096, 32, 3, 1501), (2000, 12, 12, 20000)])
def test_narrow_graphs_match_the_oracle(V, width, fan, K):
    check(narrow_graph(V, width, fan, 1, 2, 9), K)


@pytest.mark.parametrize("fan,K", [(7, 5000), (29, 3001)])
def test_forks_and_joins_match_the_oracle(fan, K):
    """A source, `fan` operators, a sink that is the next source, and so on; every edge twice."""
    edges, at = [], 0
    for _ in range(40):
        for x in range(fan):
            edges += [(at, at + 1 + x), (at + 1 + x, at + 1 + fan)] * 2
        at += fan + 1
    V = at + 1
    w = ck.problem(V, edges, np.ones(V, np.int64), 2)
    w.assign_mode, w.group = "per_op", None
    check(w, K)


@pytest.mark.parametrize("config,kw,K", [(1, {}, 1024), (3, {}, 1000), (4, {}, 2001), (4, dict(microbatches=12), 300)])
def test_pipelines_and_model_graphs_match_the_oracle(config, kw, K):
    check(wl.make_config(config, **kw), K)
