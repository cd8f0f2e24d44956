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
    for lane in (2, 0):
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


@pytest.mark.parametrize("scale,wg", [(13, 0), (21, 0), (21, 1)])
def test_lane_tier_every_batch(scale, wg):
    # the lane tier before each warp tier (2: on every batch), sets of 1 to hundreds of nodes
    g = P.ssa_gen_rmat(scale, 8 << scale, seed=3)
    P.ssa_set_tuning(g, 0)
    P.ssa_set_warp_tier(g, wg)
    got = []
    for lane in (0, 1, 2):
        P.ssa_set_lane_tier(g, lane)
        p = P.Pool(g, P.SSA_IC, 5, 3).grow(40_000)
        sizes = p.set_sizes()
        S = p.max_coverage(40_000, 20)
        est = P.ssa_estimate_inf(g, P.SSA_IC, 5, 9, S[0], 900.5, 50_000)
        got.append((p.counts(40_000), sizes, S[0], S[1], est))
        p.free()
    assert got[0][1].max() > 64
    for other in got[1:]:
        for x, y in zip(got[0], other):
            assert np.array_equal(x, y)
    g.free()
