"""IC with per-edge coins where the 4-edge groups, the 32-group slabs, the
64-group pieces of shared in-lists and the stage of live tails have their edges:
in-lists of every length around those sizes, at every alignment, rooted at
through the benefit weights, in the warp tiers and the CTA tier.  RR sets and
hit counts equal the oracle's exactly."""
import numpy as np
import pytest

import inputs
import oracle

pytestmark = pytest.mark.gpu
P = pytest.importorskip("paper_1605_07990_gb300")

DEGREES = [1, 2, 3, 4, 5, 7, 8, 9, 127, 128, 129, 130, 255, 256, 257, 511, 512, 513, 1023, 1025, 2043, 2045, 2047,
           2048, 2049, 2050, 2052, 2303, 2305, 4095, 4097, 8191, 8193]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _hubs(seed):
    # hub h has DEGREES[h] in-edges from random leaves; every leaf has a few in-edges from leaves and hubs
    rng = np.random.default_rng(seed)
    H, n = len(DEGREES), 12_289
    src = [rng.choice(np.arange(H, n), d, replace=False) for d in DEGREES]
    dst = [np.full(d, h) for h, d in enumerate(DEGREES)]
    src.append(rng.integers(0, n, 3 * n))
    dst.append(rng.integers(H, n, 3 * n))
    return inputs.EdgeList(n, np.concatenate(src).astype(np.int32), np.concatenate(dst).astype(np.int32)), H


@pytest.mark.parametrize("weights", ["trivalency", "explicit"])
@pytest.mark.parametrize("mid,heavy", [(0, 0x7FFFFFFF), (0, 1), (16384, 0x7FFFFFFF), (16384, 64)])
def test_group_edges_match_oracle(weights, mid, heavy):
    el, H = _hubs(5)
    if weights == "trivalency":
        kind, thr = oracle.W_TRIVALENCY, None
    else:
        kind = oracle.W_EXPLICIT
        thr = np.random.default_rng(6).integers(0, 2**31, el.m, dtype=np.uint64).astype(np.uint32)
        thr[::97] = 0xFFFFFFFF
        thr[::101] = 0
    og = oracle.Graph(el.n, el.src, el.dst, kind, thr, 3)
    gg = P.ssa_load_graph(el.n, el.src, el.dst, thr, kind, 3)
    for x, y in zip(og.csr(), P.ssa_graph_export(gg)):
        assert np.array_equal(x, y)
    P.ssa_set_tuning(gg, mid, heavy)
    b = np.zeros(el.n, np.uint32)
    b[:H] = 1  # every hub is a root
    N = 400
    op = oracle.Pool(og, oracle.IC, 11, 2, b).grow(N)
    gp = P.Pool(gg, P.SSA_IC, 11, 2, b).grow(N)
    for j, (x, y) in enumerate(zip(op.sets(), gp.sets())):
        assert np.array_equal(np.sort(x), y), j
    S = np.array([H + 1, H + 77, el.n - 1], np.int32)
    for lam in (20.5, 150.0):
        assert P.ssa_estimate_inf(gg, P.SSA_IC, 11, 4, S, lam, 1500, benefit=b) == \
            oracle.estimate_inf(og, oracle.IC, 11, 4, S, lam, 1500, benefit=b)[:2]
    gp.free()
    gg.free()
