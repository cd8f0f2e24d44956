"""A D-SSA round whose Max-Coverage gave up at a barrier: its seeds were never
written, and the stare behind it (in the same CUDA graph, or launched apart)
must not act on what the buffer holds.  The buffers of the small graph's solve
come out of the memory that solves of a 64 times larger graph gave back, seed
ids far outside the small graph's range among it.  Nothing waits forever: the
bound of one poll only makes the kernel return early."""
import numpy as np
import pytest

import inputs
import oracle

pytestmark = pytest.mark.gpu
P = pytest.importorskip("paper_1605_07990_gb300")
SSA_E_TIMEOUT = 5


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("captured", [False, True], ids=["apart", "captured"])
@pytest.mark.parametrize("k", [1, 600])
def test_unwritten_seeds_reach_no_memory(captured, k):
    el = inputs.rmat(14, 1 << 17, seed=1)
    n = el.n
    big = P.ssa_gen_rmat(20, 1 << 22, seed=2)
    g = P.ssa_load_graph(n, el.src, el.dst, None, P.SSA_W_WC)
    for seed in (1, 2):
        P.ssa_solve(big, P.SSA_ALGO_DSSA, P.SSA_LT, k, 0.2, 1e-6, seed)
    sv = P.Solver(g)
    sv.set_graphs(captured)
    try:
        P.ssa_set_greedy_mode(1)
        P.ssa_set_wait_polls(1)
        for seed in (3, 4):
            with pytest.raises(P.SSAError) as e:
                sv.solve(P.SSA_ALGO_DSSA, P.SSA_IC, k, 0.1, 1.0 / n, seed)
            assert e.value.status == SSA_E_TIMEOUT
    finally:
        P.ssa_set_wait_polls(0)
        P.ssa_set_greedy_mode(0)
    og = oracle.Graph(n, el.src, el.dst, oracle.W_WC)
    r = sv.solve(P.SSA_ALGO_DSSA, P.SSA_IC, k, 0.1, 1.0 / n, 3)
    o = oracle.solve(og, oracle.DSSA, oracle.IC, k, 0.1, 1.0 / n, 3)
    assert np.array_equal(r.seeds, o.seeds) and r.trace == o.trace
    sv.free()
    g.free()
    big.free()
