"""The bound on the greedy's barrier waits (ssa_set_wait_polls) is on polls
without progress: while one block makes a session's picks, thousands of them,
the others wait at one barrier for as long as the picks go on, and a bound that
spans a pick but no session does not end the call."""
import numpy as np
import pytest

import inputs
import oracle

pytestmark = pytest.mark.gpu
P = pytest.importorskip("paper_1605_07990_gb300")


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("n,sets,k", [(70_001, 200_000, 20_000), (3001, 30_000, 2500)], ids=["lists", "shared"])
def test_a_session_outlasts_the_bound(n, sets, k):
    # no edges: every set is its root, so nodes tie and a session makes thousands of picks
    el = inputs.edges(n, [])
    op = oracle.Pool(oracle.Graph(n, el.src, el.dst, oracle.W_WC), oracle.IC, 3, 0).grow(sets)
    g = P.ssa_load_graph(n, el.src, el.dst, None, P.SSA_W_WC)
    gp = P.Pool(g, P.SSA_IC, 3, 0).grow(sets)
    want = op.max_coverage(sets, k)
    try:
        P.ssa_set_greedy_mode(1)
        P.ssa_set_wait_polls(1000)  # about a millisecond; the picks take several
        got = gp.max_coverage(sets, k)
    finally:
        P.ssa_set_wait_polls(0)
        P.ssa_set_greedy_mode(0)
    assert np.array_equal(want[0], got[0]) and np.array_equal(want[1], got[1]) and want[2] == got[2]
    gp.free()
    g.free()
