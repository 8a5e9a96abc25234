"""GPU tests of the row kernels at the lengths where they change: aggregated
rows in ascending target order (deterministic mode, against the oracle's
stored CSR) and the rows of an edge list sorted and merged."""
import numpy as np
import pytest
import torch

import gen
import oracle
import paper_2312_13936_gb300 as lg
from tests._gpu import compare_traces, run_gpu

pytestmark = pytest.mark.gpu


def _spokes(k, size=3):
    """A vertex joined to one vertex of each of k cliques: once the cliques are
    communities, its row has k targets."""
    us, vs = [], []
    for q in range(k):
        b = 1 + q * size
        us += [0] + [b + i for i in range(size) for j in range(i + 1, size)]
        vs += [b] + [b + j for i in range(size) for j in range(i + 1, size)]
    order = np.random.default_rng(k).permutation(1 + k * size)  # targets in no particular order
    return gen.from_edges(1 + k * size, order[np.array(us)], order[np.array(vs)])


@pytest.mark.parametrize("k", [6, 8, 15, 31, 32, 33, 254, 256, 257, 2047, 2049, 4095, 8191, 8193, 9000])
def test_aggregated_rows_as_stored(k):
    g = _spokes(k)
    ref = oracle.leiden(g, mode=oracle.SYNC, trace=True)
    memb, q, st, tr = run_gpu(g, lg.LEIDEN_DETERMINISTIC, trace=True)
    assert not compare_traces(tr, ref.trace)
    assert np.array_equal(memb, ref.membership)


@pytest.mark.parametrize("d", [1, 7, 8, 9, 31, 32, 33, 255, 256, 257, 2047, 2048, 2049, 16383, 16384, 16385, 40000])
@pytest.mark.parametrize("combine", ["sum", "max"])
@pytest.mark.parametrize("weighted", [True, False])
def test_edge_rows_of_every_length(d, combine, weighted):
    """Vertex 0 listed with d edges (a quarter of them repeats, one a
    self-loop when d > 4) among random others."""
    rng = np.random.default_rng(d)
    n = 50000
    u = rng.integers(1, n, d).astype(np.int32)
    if d > 4:
        u[: d // 4] = u[d // 4: 2 * (d // 4)]
        u[-1] = 0
    a, b = rng.integers(0, n, 5000).astype(np.int32), rng.integers(0, n, 5000).astype(np.int32)
    src, dst = np.concatenate([np.zeros(d, np.int32), a]), np.concatenate([u, b])
    order = rng.permutation(len(src))
    src, dst = src[order], dst[order]
    w = rng.integers(1, 9, len(src)).astype(np.float32) if weighted else None
    ref = oracle.csr_from_edges(n, src, dst, w, combine=combine)
    got = lg.csr_from_edges(n, torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda(),
                            None if w is None else torch.from_numpy(w).cuda(), combine=combine)
    for x, y, what in zip(got, ref, ("offsets", "indices", "weights")):
        assert np.array_equal(x.cpu().numpy(), y), what


@pytest.mark.parametrize("d", [257, 300, 1025, 2048, 2049, 9001, 16384])
@pytest.mark.parametrize("span", [1, 40, 2000, 30000])
def test_edge_rows_of_crowded_targets(d, span):
    """Vertex 0 listed with d edges into a range of span vertices among two
    million, so that its row's targets share few of the high-bit buckets."""
    rng = np.random.default_rng(d * 7 + span)
    n = 2_000_000
    u = (1_234_567 + rng.integers(0, span, d)).astype(np.int32)
    a, b = rng.integers(0, n, 5000).astype(np.int32), rng.integers(0, n, 5000).astype(np.int32)
    src, dst = np.concatenate([np.zeros(d, np.int32), a]), np.concatenate([u, b])
    order = rng.permutation(len(src))
    src, dst = src[order], dst[order]
    w = rng.integers(1, 9, len(src)).astype(np.float32)  # sums below 2^24: exact in any order
    ref = oracle.csr_from_edges(n, src, dst, w)
    got = lg.csr_from_edges(n, torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda(), torch.from_numpy(w).cuda())
    for x, y, what in zip(got, ref, ("offsets", "indices", "weights")):
        assert np.array_equal(x.cpu().numpy(), y), what
