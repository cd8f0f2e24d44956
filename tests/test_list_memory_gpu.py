"""Device memory of Max-Coverage's candidate lists: what a kept solver holds
after a solve of millions of sets, and solves whose lists get the little that
the pool leaves of its cap, against the solve without one."""
import ctypes as C

import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu
P = pytest.importorskip("paper_1605_07990_gb300")
USED_MEM_CURRENT = 7  # cudaMemPoolAttrUsedMemCurrent


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _pool_bytes():
    """Bytes handed out by the device's default memory pool."""
    rt = C.CDLL("libcudart.so")
    pool, used = C.c_void_p(), C.c_uint64()
    assert rt.cudaDeviceSynchronize() == 0
    assert rt.cudaDeviceGetDefaultMemPool(C.byref(pool), 0) == 0
    assert rt.cudaMemPoolGetAttribute(pool, USED_MEM_CURRENT, C.byref(used)) == 0
    return used.value


def test_lists_of_a_large_solve_are_given_back():
    g = P.ssa_gen_rmat(16, 1 << 20, seed=2)
    sv = P.Solver(g)
    args = (P.SSA_ALGO_DSSA, P.SSA_IC, 20)
    sv.solve(*args, 0.3, 1.0 / g.n, 1)
    before = _pool_bytes()
    r = sv.solve(*args, 0.01, 1.0 / g.n, 1)
    held = _pool_bytes() - before
    n, e = r.trace[-1]["n_sets"], r.pool_entries
    lists = 4 * min(e, max(2 * n, 1 << 25)) + 17 * min((e + 19 * n) // 8, 1 << 25)
    # per set of a batch: six hand-over lists of 8 bytes, the hit and the covered flag
    scratch = 50 * n
    assert lists > 160 << 20
    assert held <= scratch + (80 << 20)
    sv.free()
    g.free()


@pytest.mark.parametrize("captured", [False, True], ids=["apart", "captured"])
@pytest.mark.parametrize("model", [P.SSA_IC, P.SSA_LT], ids=["ic", "lt"])
def test_lists_with_little_room(model, captured):
    el = inputs.rmat(15, 1 << 18, seed=9)
    g = P.ssa_load_graph(el.n, el.src, el.dst, None, P.SSA_W_WC)
    args = (P.SSA_ALGO_DSSA, model, 300, 0.02, 1.0 / g.n, 8)
    want = P.ssa_solve(g, *args)
    sets = want.trace[-1]["n_sets"]
    sv = P.Solver(g)
    sv.set_graphs(captured)
    need = 12 * want.pool_entries + 14 * sets
    for f in (1.0, 1.3, 4.0):
        got = sv.solve(*args, pool_bytes_cap=int(need * f) + 64)
        assert np.array_equal(got.seeds, want.seeds) and got.trace == want.trace
        assert got.influence == want.influence and got.n_rr == want.n_rr
    sv.free()
    g.free()
