"""GPU tests of rows that are split by ranges of their targets: rows of an edge
list beyond a block's shared memory among more than 2^20 vertices, more of
their parts than are taken at once, and rows of the aggregated graph beyond
8,192 entries among more than 2^18 communities."""
import numpy as np
import pytest
import torch

import oracle
import paper_2312_13936_gb300 as lg
from tests._gpu import compare_traces, run_gpu
from tests.test_gpu_rows import _spokes

pytestmark = pytest.mark.gpu


def _targets(rng, n, d, kind):
    """d targets of vertex 0: over all ranges, all within a few thousand
    vertices around a range's bound, or one range full and one target in each
    other."""
    if kind == "spread":
        return rng.integers(1, n, d)
    if kind == "crowded":
        return (1 << 20) - 2000 + rng.integers(0, 4000, d) % (n - (1 << 20) + 2000)
    u = rng.integers(1, 1 << 20, d)
    u[: n >> 20] = np.minimum(n - 1, (np.arange(n >> 20) + 1) << 20)
    return u


@pytest.mark.parametrize("n", [1 << 20, (1 << 20) + 1, 3 * (1 << 20) + 5])
@pytest.mark.parametrize("d", [16385, 40000, 300000])
@pytest.mark.parametrize("kind", ["spread", "crowded", "one_range"])
@pytest.mark.parametrize("weighted,combine", [(False, "sum"), (True, "sum"), (True, "max")])
def test_edge_rows_by_ranges(n, d, kind, weighted, combine):
    rng = np.random.default_rng(d + n)
    u = _targets(rng, n, d, kind)
    a, b = rng.integers(0, n, 5000), rng.integers(0, n, 5000)
    src = np.concatenate([np.zeros(d), a]).astype(np.int32)
    dst = np.concatenate([u, b]).astype(np.int32)
    order = rng.permutation(len(src))
    src, dst = src[order], dst[order]
    w = rng.integers(1, 9, len(src)).astype(np.float32) if weighted else None  # sums below 2^24: exact in any order
    ref = oracle.csr_from_edges(n, src, dst, w, combine=combine)
    got = lg.csr_from_edges(n, torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda(),
                            None if w is None else torch.from_numpy(w).cuda(), combine=combine)
    for x, y, what in zip(got, ref, ("offsets", "indices", "weights")):
        assert np.array_equal(x.cpu().numpy(), y), what


@pytest.mark.parametrize("n", [1 << 20, (1 << 20) + 3000])
def test_more_long_parts_than_at_once(n):
    """8,200 rows of 16,500 entries in one range: their bitmaps are taken in
    two waves. Against torch's sort and merge of the keys."""
    rows, d = 8200, 16500
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    src = torch.arange(rows, device="cuda").repeat_interleave(d)
    dst = torch.randint(rows, 1 << 20, (rows * d,), device="cuda", generator=g)
    if n > 1 << 20:  # a few targets in the second range
        dst[::5000] = torch.randint(1 << 20, n, (dst[::5000].numel(),), device="cuda", generator=g)
    off, idx, w = lg.csr_from_edges(n, src.int(), dst.int())
    key, count = torch.unique(src * n + dst, return_counts=True)  # src < dst: no edge is listed both ways round
    key, order = torch.sort(torch.cat([key, key % n * n + key // n]))
    count = torch.cat([count, count])[order]
    want = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    want[1:] = torch.cumsum(torch.bincount(key // n, minlength=n), 0)
    assert torch.equal(off, want)
    assert torch.equal(idx.long(), key % n)
    assert torch.equal(w.long(), count)


def test_aggregated_row_by_ranges():
    """A vertex joined to 262,500 cliques: its row as a super-vertex has a full
    range of 2^18 communities and one of a few hundred."""
    g = _spokes(262_500)
    ref = oracle.leiden(g, mode=oracle.SYNC, trace=True)
    memb, _, _, tr = run_gpu(g, lg.LEIDEN_DETERMINISTIC, trace=True)
    assert max(int(t[lg.TRACE_AGG_DEG].max()) for t in tr.values() if lg.TRACE_AGG_DEG in t) > 262_144
    assert not compare_traces(tr, ref.trace)
    assert np.array_equal(memb, ref.membership)
