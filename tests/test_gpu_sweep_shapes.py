"""GPU tests of the persistent sweep's work division: graphs at the edges of
its rules (one block or many, units of 2, 8 or 32 vertices in the apply phase,
rows at the flat walk's bound, the bins' bounds) against the oracle's SYNC
mode, bit for bit."""
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


@pytest.mark.parametrize("n", [1, 2, 31, 33, 500, 1023, 1025, 1537, 4999, 40001])
def test_sizes_around_one_block(n):
    _equal(gen.sbm(n, max(1, n // 100), 0.1 if n < 2000 else 200.0 / n, 1.0 / n, seed=n))


@pytest.mark.parametrize("d", [8, 9, 16, 17, 32, 33, 256, 257, 1023, 1024, 1025, 2048, 2049, 5000])
@pytest.mark.parametrize("hubs", [1, 5])
def test_row_lengths(d, hubs):
    _equal(_star(d, hubs))
