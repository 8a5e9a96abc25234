"""GPU tests of batches and served unions whose weights add up beyond 63 bits
while every graph keeps the deterministic mode's 2m < 2^53 (the rule holds per
graph): each graph against the oracle's SYNC mode, as it comes out alone."""
import numpy as np
import pytest

import gen
import oracle
import paper_2312_13936_gb300 as lg

pytestmark = pytest.mark.gpu


# 2m together 2^63, 2^64, and just above 2^63 with the largest 2m that one
# graph can have (weights exact in fp32)
@pytest.mark.parametrize("graphs,weight", [(2048, 2.0**51), (4096, 2.0**51), (1026, 2.0**52 - 2.0**28)])
@pytest.mark.parametrize("served", [False, True])
def test_weight_sums_beyond_63_bits(graphs, weight, served):
    pair = gen.from_edges(2, [0], [1], [weight])
    ref = oracle.leiden(pair, mode=oracle.SYNC)
    assert np.array_equal(ref.membership, [0, 0])
    want = np.tile(ref.membership, graphs)
    if served:
        srv = lg.LeidenServer(2 * graphs, 2 * graphs, max_graphs=graphs, mode=lg.LEIDEN_DETERMINISTIC)
        try:
            for _ in range(graphs):
                srv.submit(pair.offsets, pair.indices, pair.weights)
            done = []
            while len(done) < graphs:
                srv.step()
                done += srv.results()
        finally:
            srv.close()
        done.sort(key=lambda r: r[0])
        memb, q = np.concatenate([r[1] for r in done]), np.array([r[2] for r in done])
    else:
        h = lg.LeidenBatch(*lg.pack_batch([pair] * graphs))
        try:
            memb, q, _ = h.run(mode=lg.LEIDEN_DETERMINISTIC)
            memb = memb.cpu().numpy()
        finally:
            h.close()
    assert np.array_equal(memb, want)
    assert np.all(np.abs(q - ref.modularity) <= 1e-9)
