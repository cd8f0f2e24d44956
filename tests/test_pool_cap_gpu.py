"""Byte caps of the RR pool (ssa_params.pool_bytes_cap): a solve whose pool fits
its cap gives the answer it gives without one, however near the cap is, and one
whose pool does not fit reports SSA_E_POOL_FULL.  The pool takes 12 bytes an
entry and 14 a set."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu
P = pytest.importorskip("paper_1605_07990_gb300")
SSA_E_POOL_FULL = 3


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _graph(weights):
    el = inputs.rmat(16, 1 << 19, seed=4)
    if weights == "wc":
        return P.ssa_load_graph(el.n, el.src, el.dst, None, P.SSA_W_WC)
    d = np.bincount(el.dst, minlength=el.n)  # the same in-weights, edge by edge
    thr = ((1 << 32) // np.maximum(d, 2))[el.dst].astype(np.uint32)
    return P.ssa_load_graph(el.n, el.src, el.dst, thr, P.SSA_W_EXPLICIT)


@pytest.mark.parametrize("weights,model", [("wc", P.SSA_IC), ("explicit", P.SSA_IC), ("wc", P.SSA_LT)])
def test_solve_within_its_cap(weights, model):
    g = _graph(weights)
    args = (P.SSA_ALGO_DSSA, model, 40, 0.05, 1.0 / g.n, 6)
    want = P.ssa_solve(g, *args)
    sets = want.trace[-1]["n_sets"]
    assert want.n_rr == 2 * sets > 50_000
    need = 12 * want.pool_entries + 14 * sets
    sv = P.Solver(g)
    for f in (1.5, 1.2, 1.1, 1.01):
        got = sv.solve(*args, pool_bytes_cap=int(need * f))
        assert np.array_equal(got.seeds, want.seeds) and got.trace == want.trace
        assert got.pool_entries == want.pool_entries and got.influence == want.influence
    with pytest.raises(P.SSAError) as e:
        sv.solve(*args, pool_bytes_cap=int(need * 0.6))
    assert e.value.status == SSA_E_POOL_FULL
    got = sv.solve(*args, pool_bytes_cap=int(need * 1.1))
    assert np.array_equal(got.seeds, want.seeds) and got.trace == want.trace
    sv.free()
    g.free()
