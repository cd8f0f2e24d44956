"""ssa_coverage_noalloc over arrays of every alignment and length around its
16-byte loads, exactly against a plain count: slices that start off a 16-byte
boundary go entry by entry, and the last entries of a vector pass are its tail."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("node_at,samp_at", [(0, 0), (1, 1), (0, 3), (2, 0), (4, 8)])
@pytest.mark.parametrize("entries", [0, 1, 3, 4, 5, 1023, 4097, 700_001])
def test_alignment_and_tails(node_at, samp_at, entries):
    torch = pytest.importorskip("torch")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1605_07990_gb300 as P

    rng = np.random.default_rng(entries + node_at)
    n, sets, first, count = 5003, max(1, entries // 7), 1, max(1, entries // 9)
    nodes = rng.integers(0, n, entries).astype(np.int32)
    samp = rng.integers(0, sets, entries).astype(np.int32)
    seeds = rng.choice(n, 40, replace=False).astype(np.int32)
    inside = (samp >= first) & (samp < first + count)
    want = len(np.unique(samp[inside & np.isin(nodes, seeds)]))
    a = torch.zeros(entries + 16, dtype=torch.int32, device="cuda")
    b = torch.zeros(entries + 16, dtype=torch.int32, device="cuda")
    a[node_at:node_at + entries] = torch.from_numpy(nodes).cuda()
    b[samp_at:samp_at + entries] = torch.from_numpy(samp).cuda()
    s = torch.from_numpy(seeds).cuda()
    stream = torch.cuda.current_stream().cuda_stream
    got = P.ssa_coverage_noalloc(n, a[node_at:].data_ptr(), b[samp_at:].data_ptr(), entries, first, count,
                                 s.data_ptr(), len(seeds), stream)
    assert got == want
