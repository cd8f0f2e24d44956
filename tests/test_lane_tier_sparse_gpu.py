"""The lane tier's rule on graphs whose visited set fits shared memory: a large
batch of sets of a few nodes (a sparse graph) goes through it, one of larger sets
and a small batch do not.  What shows it are the in-edges that the tier looked at
before it handed a large set on; the sets are the same."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
P = pytest.importorskip("paper_1605_07990_gb300")


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("degree,sets,takes", [(1, 280_000, True), (16, 280_000, False), (1, 200_000, False)])
def test_rule_follows_the_sets(degree, sets, takes):
    g = P.ssa_gen_rmat(14, degree << 14, seed=3)
    got = {}
    for on in (-1, 0, 1):
        P.ssa_set_lane_tier(g, on)
        p = P.Pool(g, P.SSA_IC, 5, 0)
        p.grow(2048)  # the rule knows these sets when it meets the large batch
        got[on] = (p.grow(sets).info(), p.counts(sets))
        p.free()
    assert all(x[0][:2] == got[0][0][:2] and np.array_equal(x[1], got[0][1]) for x in got.values())
    assert got[0][0][2] < got[1][0][2]
    assert (got[-1][0][2] > got[0][0][2]) == takes
    g.free()
