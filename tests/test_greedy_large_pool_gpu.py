"""Max-Coverage over more sets than candidate lists with room for every member
hold (2^25 chunks): the picks against a closed form.  The graph is one path
0 -> 1 -> ... with p = 1 (the set of v is {0, ..., v}: long sets) and pairs
a -> a + 1 with p = 1, so that node 0 and the first node of each pair cover
their parts whole, and the picks are those by (count, smaller id)."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu
P = pytest.importorskip("paper_1605_07990_gb300")


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("sets", [16_000_001, 21_000_003])  # below and above the room
def test_more_sets_than_lists_hold(sets, mode):
    n, path, k = 1 << 18, 600, 400
    el = inputs.edges(n, [(v, v + 1) for v in range(path - 1)] + [(a, a + 1) for a in range(path, n - 1, 2)])
    g = P.ssa_load_graph(el.n, el.src, el.dst, None, P.SSA_W_WC)
    P.ssa_set_greedy_mode(mode)
    try:
        p = P.Pool(g, P.SSA_IC, 5).grow(sets)
        seeds, gains, cov = p.max_coverage(sets, k)
        counts = np.asarray(p.counts(sets)).astype(np.int64)
        p.free()
    finally:
        P.ssa_set_greedy_mode(0)
    heads = np.concatenate([[0], np.arange(path, n, 2)])
    order = heads[np.lexsort((heads, -counts[heads]))][:k]
    assert np.array_equal(seeds, order)
    assert np.array_equal(gains, counts[order])
    assert cov == counts[order].sum()
    g.free()
