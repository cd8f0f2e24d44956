"""WRIS roots from prefix sums made on the device, exactly the oracle's: node
counts around the 4096-weight tiles, weights up to 2^32 - 1 (sums past 32 bits),
zero weights at the ends and a single node that holds them all.  On a graph
without edges an RR set is its root."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
P = pytest.importorskip("paper_1605_07990_gb300")


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("n", [1, 2, 3, 4095, 4096, 4097, 8191, 40_961, 300_007])
@pytest.mark.parametrize("kind", ["large", "zeros", "one"])
def test_roots_match_oracle(n, kind):
    rng = np.random.default_rng(n)
    b = rng.integers(0, 2**32, n, dtype=np.uint64).astype(np.uint32)
    if kind == "zeros":
        b[: n // 3] = 0
        b[n - n // 4:] = 0
        b[n // 3] = 5
    if kind == "one":
        b[:] = 0
        b[n - 1] = 1
    if int(b.sum(dtype=np.uint64)) == 0:
        b[0] = 1
    none = np.zeros(0, np.int32)
    og = oracle.Graph(n, none, none, oracle.W_WC)
    gg = P.ssa_load_graph(n, none, none)
    N = 5000
    op = oracle.Pool(og, oracle.IC, 3, 7, b).grow(N)
    gp = P.Pool(gg, P.SSA_IC, 3, 7, b).grow(N)
    assert np.array_equal(op.counts(N), gp.counts(N).astype(np.int64))
    assert [int(x[0]) for x in op.sets()[:500]] == [int(x[0]) for x in gp.sets(0, 500)]
    gp.free()
    with pytest.raises(P.SSAError):
        P.Pool(gg, P.SSA_IC, 3, 7, np.zeros(n, np.uint32))
    gg.free()
