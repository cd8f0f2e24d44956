"""ssa_set_lane_tier: on > 0 runs the lane tier on every batch, 0 on none, < 0 by
the rule of a new graph.  The sets are the same; what tells the settings apart is
the in-edges that the lane tier looked at before it handed a large set on."""
import pytest

pytestmark = pytest.mark.gpu
P = pytest.importorskip("paper_1605_07990_gb300")


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def test_one_asks_for_it_on_every_batch():
    g = P.ssa_gen_rmat(13, 1 << 17, seed=3)  # warps with their visited set in shared memory: not by the rule

    def visits(on):
        if on is not None:
            P.ssa_set_lane_tier(g, on)
        p = P.Pool(g, P.SSA_IC, 5, 0).grow(1000)
        sets, entries, edges = p.info()
        p.free()
        return sets, entries, edges

    new, never, one, two, rule = (visits(on) for on in (None, 0, 1, 2, -1))
    assert new == never == rule and one == two
    assert one[:2] == never[:2] and one[2] > never[2]
    g.free()
