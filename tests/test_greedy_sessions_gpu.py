"""Max-Coverage (Algorithm 2) where its sessions can go wrong, against the
oracle (exact): gains past what a session's keys hold, more ties than a session
has candidates, sets at the length where their lists are shared between warps,
member counts around the chunks of a list, and pools of no, one and few sets,
under each launch shape."""
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


def _star(n):  # every set holds node 0
    return inputs.edges(n, [(0, v) for v in range(1, n)])


def _path(n):  # with p = 1 the set of v is {0, ..., v}: every length up to n
    return inputs.edges(n, [(v, v + 1) for v in range(n - 1)])


def _combs(teeth, length):  # disjoint paths: sets of every length, no shared hub
    return inputs.edges(teeth * length, [(t * length + i, t * length + i + 1) for t in range(teeth)
                                         for i in range(length - 1)])


CASES = {
    # name: edge list, sets, picks
    "wide_gains": (_star(1001), 270_000, (1, 40)),        # first gain 270,000 > 2^18
    "ties": (inputs.edges(70_001, []), 200_000, (30, 20_000)),
    "long_sets": (_path(701), 3000, (1, 9, 701)),
    "chunk_edges": (_combs(40, 70), 4000, (60, 2800)),
    "no_sets": (_path(33), 0, (1, 33)),
    "one_set": (_path(5), 1, (5,)),
    "few": (_combs(3, 11), 64, (1, 33)),
}


@pytest.mark.parametrize("mode", [0, 1, 2], ids=["auto", "grid", "cluster"])
@pytest.mark.parametrize("name", sorted(CASES))
def test_sessions_match_oracle(name, mode):
    el, N, ks = CASES[name]
    thr = np.full(el.m, 0xFFFFFFFF, np.uint32)
    og = oracle.Graph(el.n, el.src, el.dst, oracle.W_EXPLICIT, thr, 1)
    gg = P.ssa_load_graph(el.n, el.src, el.dst, thr, P.SSA_W_EXPLICIT, 1)
    op = oracle.Pool(og, oracle.IC, 3, 0).grow(N)
    gp = P.Pool(gg, P.SSA_IC, 3, 0).grow(N)
    P.ssa_set_greedy_mode(mode)
    try:
        # a cut inside the pool first, then all of it: the counts go on, then start over
        for cut in (N - N // 3, N, N // 2):
            assert np.array_equal(op.counts(cut), gp.counts(cut).astype(np.int64))
            for k in ks:
                want, got = op.max_coverage(cut, k), gp.max_coverage(cut, k)
                assert np.array_equal(want[0], got[0]) and np.array_equal(want[1], got[1]) and want[2] == got[2]
    finally:
        P.ssa_set_greedy_mode(0)
    gp.free()
    gg.free()
