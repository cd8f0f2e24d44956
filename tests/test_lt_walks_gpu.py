"""LT walks where their tiers and searches have their edges, against the oracle,
exactly: walks of a few to 1500 nodes (past the warp tier's list), and in-lists of
general in-weights of every length around the 8-way and 33-way searches and the
thread, warp and block sums, with zero thresholds, sums of exactly 2^32 and
sums short of it."""
import numpy as np
import pytest

import inputs
import oracle

pytestmark = pytest.mark.gpu
P = pytest.importorskip("paper_1605_07990_gb300")

DEGREES = [1, 2, 7, 8, 9, 16, 17, 31, 32, 33, 34, 63, 65, 71, 257, 1056, 1057, 1089, 1090, 4095, 4096, 4097, 9001]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _check(og, gg, seed, N, benefit=None):
    op = oracle.Pool(og, oracle.LT, seed, 1, benefit).grow(N)
    gp = P.Pool(gg, P.SSA_LT, seed, 1, benefit).grow(N)
    assert np.array_equal(op.counts(N), gp.counts(N).astype(np.int64))
    for j, (x, y) in enumerate(zip(op.sets()[:3000], gp.sets(0, min(N, 3000)))):
        assert np.array_equal(np.sort(x), y), j
    S = op.max_coverage(N, 3)[0]
    for need in (10.5, 0.7 * N):
        assert P.ssa_estimate_inf(gg, P.SSA_LT, seed, 2, S, need, 3 * N, benefit=benefit) == \
            oracle.estimate_inf(og, oracle.LT, seed, 2, S, need, 3 * N, benefit=benefit)[:2]
    gp.free()


@pytest.mark.parametrize("N", [500, 20_000])
@pytest.mark.parametrize("explicit", [False, True])
def test_walk_lengths(N, explicit):
    # a ring of 1500 nodes with a few chords: walks of a few to 1500 nodes
    n = 1500
    rng = np.random.default_rng(2)
    src = np.concatenate([np.arange(n), rng.integers(0, n, 12)]).astype(np.int32)
    dst = np.concatenate([(np.arange(n) + 1) % n, rng.integers(0, n, 12)]).astype(np.int32)
    kind, thr = oracle.W_WC, None
    if explicit:
        kind = oracle.W_EXPLICIT
        deg = np.bincount(dst, minlength=n)[dst]
        thr = np.minimum((0.985 * 2.0**32 / deg).astype(np.uint64), 2**32 - 1).astype(np.uint32)
    og = oracle.Graph(n, src, dst, kind, thr, 1)
    gg = P.ssa_load_graph(n, src, dst, thr, kind, 1)
    _check(og, gg, 5, N)
    gg.free()


@pytest.mark.parametrize("N", [3000, 20_000])
def test_search_lengths(N):
    rng = np.random.default_rng(4)
    H, n = len(DEGREES), 10_007
    src = [rng.choice(np.arange(H, n), d, replace=False) for d in DEGREES]
    dst = [np.full(d, h) for h, d in enumerate(DEGREES)]
    src.append(rng.integers(0, n, n))  # leaves lead on to hubs and leaves
    dst.append(rng.integers(H, n, n))
    src, dst = np.concatenate(src).astype(np.int32), np.concatenate(dst).astype(np.int32)
    w = rng.integers(0, 1000, src.size).astype(np.float64)
    w[rng.random(src.size) < 0.1] = 0
    tot = np.bincount(dst, weights=w, minlength=n)
    share = np.where(np.arange(n) % 3 == 0, 1.0, rng.uniform(0.3, 1.0, n))
    thr = np.minimum(np.floor(w * (share / np.maximum(tot, 1))[dst] * 2.0**32), 2**32 - 1).astype(np.uint64)
    order = np.lexsort((src, dst))
    for h in range(0, H, 3):  # sums of exactly 2^32: what floor left goes to the last edge of the list
        e = order[dst[order] == h]
        rest = 2**32 - int(thr[e].sum())
        thr[e[-1]] = min(int(thr[e[-1]]) + rest, 2**32 - 1)
    og = oracle.Graph(n, src, dst, oracle.W_EXPLICIT, thr.astype(np.uint32), 1)
    gg = P.ssa_load_graph(n, src, dst, thr.astype(np.uint32), P.SSA_W_EXPLICIT, 1)
    b = np.ones(n, np.uint32)
    b[:H] = 400
    _check(og, gg, 7, N, b)
    gg.free()
