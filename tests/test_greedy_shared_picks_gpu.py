"""Max-Coverage picks whose lists are so long that every block covers a share of
them (4,096 sets and more of pools of 2^23 entries and more), against the oracle
(exact): sets that overlap under many heavy picks, sets that one pick covers
whole, lists of just under and over that length, picks of more sets than a
session's keys hold, under each launch shape."""
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


def _teeth(teeth, length):  # disjoint paths with p = 1: the set of a node is the path up to it
    return inputs.edges(teeth * length, [(t * length + i, t * length + i + 1) for t in range(teeth)
                                         for i in range(length - 1)])


CASES = {
    # name: edges, weighting, model, sets, picks
    "lt_overlap": (inputs.rmat(12, 1 << 15, seed=5), oracle.W_WC, oracle.LT, 700_000, (1, 2, 40, 400)),
    "ic_overlap": (inputs.rmat(13, 1 << 17, seed=6), oracle.W_WC, oracle.IC, 1_200_000, (30, 300)),
    "whole": (_teeth(24, 50), oracle.W_EXPLICIT, oracle.IC, 500_000, (23, 24, 25, 1200)),
    "threshold": (_teeth(147, 40), oracle.W_EXPLICIT, oracle.IC, 602_000, (60, 147)),  # about 4,095 sets a tooth
    # several picks of more sets (2^18) than a session's keys hold
    "wide": (_teeth(6, 8), oracle.W_EXPLICIT, oracle.IC, 2_900_003, (5, 6, 48)),
    "wide_overlap": (inputs.rmat(9, 1 << 12, seed=5), oracle.W_WC, oracle.LT, 2_500_001, (2, 3, 30)),
}


@pytest.mark.parametrize("mode", [0, 1, 2], ids=["auto", "grid", "cluster"])
@pytest.mark.parametrize("name", sorted(CASES))
def test_shared_picks_match_oracle(name, mode):
    el, weighting, model, N, ks = CASES[name]
    thr = np.full(el.m, 0xFFFFFFFF, np.uint32) if weighting == oracle.W_EXPLICIT else None
    og = oracle.Graph(el.n, el.src, el.dst, weighting, thr, 1)
    gg = P.ssa_load_graph(el.n, el.src, el.dst, thr, weighting, 1)
    op = oracle.Pool(og, model, 3, 0).grow(N)
    gp = P.Pool(gg, model, 3, 0).grow(N)
    assert gp.info()[1] >= 1 << 23
    P.ssa_set_greedy_mode(mode)
    try:
        for cut in (N, N - N // 8):
            for k in ks:
                want, got = op.max_coverage(cut, k), gp.max_coverage(cut, k)
                assert np.array_equal(want[0], got[0]) and np.array_equal(want[1], got[1]) and want[2] == got[2]
    finally:
        P.ssa_set_greedy_mode(0)
    gp.free()
    gg.free()
