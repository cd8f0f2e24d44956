"""LT's running sums of a graph with explicit in-weights are made when its first
LT sampler starts: samplers of both models that start at the same time on several
threads share one copy and give the sets they give alone."""
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu
P = pytest.importorskip("paper_1605_07990_gb300")


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def test_first_samplers_on_several_threads():
    el = inputs.rmat(13, 1 << 16, seed=12)
    d = np.bincount(el.dst, minlength=el.n)
    thr = ((1 << 32) // np.maximum(d, 2))[el.dst].astype(np.uint32)

    def counts(g, model):
        p = P.Pool(g, model, 6, 0).grow(3000)
        c = p.counts(3000)
        p.free()
        return c

    def load():
        return P.ssa_load_graph(el.n, el.src, el.dst, thr, P.SSA_W_EXPLICIT)

    g = load()
    want = {m: counts(g, m) for m in (P.SSA_IC, P.SSA_LT)}
    held = P.ssa_graph_info(g)[2]
    g.free()
    for _ in range(4):
        g = load()
        models = [P.SSA_LT, P.SSA_IC] * 4
        with ThreadPoolExecutor(8) as ex:
            for m, c in zip(models, ex.map(lambda m: counts(g, m), models)):
                assert np.array_equal(c, want[m])
        assert P.ssa_graph_info(g)[2] == held
        g.free()
