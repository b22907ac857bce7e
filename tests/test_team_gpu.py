"""The block-per-candidate kernel where the order ends inside a window of 32 positions: the lanes beyond the end must
leave no trace in the results, whichever operator their loads fall back to.  Integers: bit-exact against the oracle."""
import numpy as np
import pytest

from paper_2503_09357_b200 import workloads as wl
from tests import checkers as ck
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


def reversed_graph(V, indeg, L):
    """Operator 0 is the last of a chain over all operators and has `indeg` sources far ahead of it in the order; every
    edge into it is far longer to communicate than the whole schedule takes."""
    edges = [(i + 1, i) for i in range(V - 1)] + [(V - 1 - q, 0) for q in range(indeg - 1)]
    comm = np.ones((len(edges), L), np.int32)
    comm[[b for b, (_, i) in enumerate(edges) if i == 0]] = 50000
    D = 3
    w = ck.problem(V, edges, np.ones(V, np.int32), D, comm=comm, L=L,
                   link_class=None if L == 1 else np.arange(D * D).reshape(D, D) % 2)
    w.assign_mode, w.group = "per_op", None
    return w


@pytest.mark.parametrize("L", [1, 2])
@pytest.mark.parametrize("indeg", [1, 3, 8])
@pytest.mark.parametrize("V", [33, 40, 63, 64, 65, 193])
def test_lanes_beyond_the_order_leave_no_trace(V, indeg, L):
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2503_09357_b200 import binding as pe
    w = reversed_graph(V, indeg, L)
    g = pe.Graph(w)
    try:
        # few candidates: six warps a block; 1000: two (the classification of a source differs)
        for K in (1, 7, 1000):
            _, order = wl.make_candidates(w, K=K)
            assign = np.ones((V, K), np.uint8)             # one machine, not machine 0: no delay applies
            for flags in (0, pe.PE_VARIANT_TEAM, pe.PE_VARIANT_TEAM | pe.PE_ASSIGN_BY_POS):
                gpu, _ = gu.check(g, w, assign, order, flags=flags, label=f"K {K} flags {flags}")
                assert (gpu["makespan"] == V).all()
    finally:
        g.close()
