"""GPU tests of the persistent sweep's work division: graphs at the edges of
its rules (one block or many, units of 2, 8 or 32 vertices in the apply phase,
rows at the flat walk's bound, the bins' bounds, the weight sum up to which
keys are 64 bits wide) against the oracle's SYNC mode, bit for bit."""
import numpy as np
import pytest

import gen
import oracle
import paper_2312_13936_gb300 as lg

pytestmark = pytest.mark.gpu


def _star(d, hubs=1):
    """hubs stars of d leaves whose leaves form one ring: rows of exactly d
    entries (the hubs) beside rows of three."""
    us, vs = [], []
    for h in range(hubs):
        base = hubs + h * d
        for k in range(d):
            us += [h, base + k]
            vs += [base + k, hubs + (base - hubs + k + 1) % (hubs * d)]
    return gen.from_edges(hubs + hubs * d, us, vs)


def _equal(g, **kw):
    ref = oracle.leiden(g, mode=oracle.SYNC, **kw)
    h = lg.Leiden(g.offsets, g.indices, g.weights)
    try:
        for _ in range(2):
            memb, q, st = h.run(mode=lg.LEIDEN_DETERMINISTIC, **kw)
            assert np.array_equal(memb.cpu().numpy(), ref.membership)
            assert abs(q - ref.modularity) <= 1e-9 * max(1.0, abs(ref.modularity))
    finally:
        h.close()


@pytest.mark.parametrize("n", [1, 2, 31, 33, 500, 1023, 1025, 1537, 4095, 4097, 4999, 40001])
def test_sizes_around_one_block(n):
    _equal(gen.sbm(n, max(1, n // 100), 0.1 if n < 2000 else 200.0 / n, 1.0 / n, seed=n))


@pytest.mark.parametrize("d", [8, 9, 16, 17, 32, 33, 256, 257, 1023, 1024, 1025, 2048, 2049, 4096, 4097, 9000])
@pytest.mark.parametrize("hubs", [1, 5])
def test_row_lengths(d, hubs):
    _equal(_star(d, hubs))


@pytest.mark.parametrize("over", [-2, 0, 2])
def test_weight_sums_around_the_narrow_arithmetic(over):
    """2m two below, at and two above 2^31 (each weight exact in fp32)."""
    g = gen.sbm(600, 6, 0.1, 0.01, seed=5)
    row = np.repeat(np.arange(g.n), np.diff(g.offsets))
    w = np.full(g.nnz, float((1 << 31) // g.nnz & ~63), np.float32)
    gap = (1 << 31) + over - int(w.astype(np.int64).sum())  # even, spread over pairs of entries
    for v in range(g.n):
        if gap == 0:
            break
        for e in range(g.offsets[v], g.offsets[v + 1]):
            u = g.indices[e]
            if u <= v or gap == 0:
                continue
            add = min(gap // 2, 1 << 20)
            back = g.offsets[u] + int(np.searchsorted(g.indices[g.offsets[u]:g.offsets[u + 1]], v))
            assert g.indices[back] == v and row[back] == u
            w[e] += add
            w[back] += add
            gap -= 2 * add
    assert gap == 0 and int(w.astype(np.int64).sum()) == (1 << 31) + over
    _equal(gen.CSR(g.n, g.offsets, g.indices, w))
