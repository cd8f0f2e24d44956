"""Weighted-cascade gaps on the GPU against the oracle, exactly: the 32-bit
logarithm decides most gaps and the exact 64-bit form the rest (none of the
small in-degrees', a third of the largest ones'), and in-degrees from 2^20 on go
by the exact form alone.  Stars whose centre is every set's source draw whole
in-lists of one in-degree."""
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


@pytest.mark.parametrize("d", [1, 2, 3, 5, 31, 100, 4095, 65_536, (1 << 17) + 1, 1 << 18, (1 << 19) + 3,
                               (1 << 20) - 1, 1 << 20, (1 << 20) + 1])
def test_star_in_lists_match_oracle(d):
    el = inputs.EdgeList(d + 1, np.arange(1, d + 1, dtype=np.int32), np.zeros(d, np.int32))
    og = oracle.Graph(el.n, el.src, el.dst, oracle.W_WC)
    gg = P.ssa_load_graph(el.n, el.src, el.dst, None, P.SSA_W_WC)
    b = np.zeros(el.n, np.uint32)
    b[0] = 1
    N = 20_000
    for lane in (1, 0):
        P.ssa_set_lane_tier(gg, lane)
        for seed, stream in ((9, 0), ((1 << 40) + 5, 255)):
            op = oracle.Pool(og, oracle.IC, seed, stream, b).grow(N)
            gp = P.Pool(gg, P.SSA_IC, seed, stream, b).grow(N)
            assert np.array_equal(op.counts(N), gp.counts(N).astype(np.int64))
            for x, y in zip(op.sets()[:400], gp.sets(0, 400)):
                assert np.array_equal(np.sort(x), y)
            gp.free()
    P.ssa_set_lane_tier(gg, 1)
    gg.free()
