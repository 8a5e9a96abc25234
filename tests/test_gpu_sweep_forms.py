"""GPU tests of the persistent sweep's compiled forms: one and two blocks per
SM (leiden_tuning.coop_blocks_per_sm; by itself a sweep takes two only with
thousands of units a step), and the deterministic mode's narrow and wide
arithmetic (2m below and from 2^31: the same graph with its weights times
2^28, exact in fp32). Deterministic runs against the oracle's SYNC mode, bit
for bit; asynchronous ones against the lower of its scores."""
import functools

import numpy as np
import pytest

import gen
import oracle
import paper_2312_13936_gb300 as lg
from tests.test_gpu_parity import hub_graph
from tests.test_gpu_sweep_shapes import _star

pytestmark = pytest.mark.gpu

# graphs whose two-block launch has more blocks than SMs: over 39,000 vertices
# at 256 a block, or rows of more than 4,096 entries, which take the whole grid
GRAPHS = {"road": lambda: gen.road(220), "sbm": lambda: gen.sbm(45000, 90, 0.1, 2e-5, seed=3),
          "rmat": lambda: gen.rmat(16, 12, seed=4), "hub_1": lambda: _star(4097), "hub_5": lambda: _star(9000, 5)}
SHAPES = {1: {"coop_blocks_per_sm": 1}, 2: {"coop_blocks_per_sm": 2, "vertices_per_block": 256}}
WIDE = 2.0**28


@functools.lru_cache(maxsize=None)
def _reference(name, scale):
    g = (GRAPHS[name] if name in GRAPHS else SMALL[name])()
    g = gen.CSR(g.n, g.offsets, g.indices, (g.weights * np.float32(scale)).astype(np.float32))
    return g, oracle.leiden(g, mode=oracle.SYNC)


# rows of every bin below the whole grid's, which the wide arithmetic meets
SMALL = {f"star_{d}": functools.partial(_star, d, 3) for d in (8, 16, 32, 33, 256, 257, 1025, 2048, 2049, 4096)}
SMALL["hubs"] = hub_graph
SMALL["rmat_12"] = lambda: gen.rmat(12, 16)


def _check_det(name, scale, tuning):
    g, ref = _reference(name, scale)
    assert (float(g.weights.astype(np.float64).sum()) >= 2.0**31) == (scale > 1)
    h = lg.Leiden(g.offsets, g.indices, g.weights, tuning=tuning)
    try:
        for _ in range(2):
            memb, q, _ = h.run(mode=lg.LEIDEN_DETERMINISTIC)
            assert np.array_equal(memb.cpu().numpy(), ref.membership)
            assert abs(q - ref.modularity) <= 1e-9 * max(1.0, abs(ref.modularity))
    finally:
        h.close()


@pytest.mark.parametrize("scale", [1.0, WIDE])
@pytest.mark.parametrize("blocks", sorted(SHAPES))
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_forms_deterministic(name, blocks, scale):
    _check_det(name, scale, SHAPES[blocks])


@pytest.mark.parametrize("name", sorted(SMALL))
def test_wide_rows_deterministic(name):
    _check_det(name, WIDE, None)


@pytest.mark.parametrize("blocks", sorted(SHAPES))
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_forms_asynchronous(name, blocks):
    g, ref = _reference(name, 1.0)
    h = lg.Leiden(g.offsets, g.indices, g.weights, tuning=SHAPES[blocks])
    try:
        memb, q, _ = h.run()
        memb = memb.cpu().numpy()
    finally:
        h.close()
    assert oracle.disconnected(g, memb)[0] == 0
    assert abs(q - oracle.modularity(g, memb)) <= 1e-9 * max(1.0, abs(q))
    assert q >= min(ref.modularity, oracle.leiden(g, mode=oracle.SEQ).modularity) - 0.01


@pytest.mark.parametrize("scale", [1.0, WIDE])
@pytest.mark.parametrize("blocks", sorted(SHAPES))
def test_forms_in_a_batch(blocks, scale):
    """40,000 vertices in all, a graph with whole-grid rows among them."""
    b = gen.sbm_batch(20, seed=17, nmin=800, nmax=5000)
    graphs = [b.graph(k) for k in range(b.num_graphs)] + [_star(4500)]
    graphs = [gen.CSR(g.n, g.offsets, g.indices, (g.weights * np.float32(scale)).astype(np.float32)) for g in graphs]
    vseg, off, idx, w = lg.pack_batch(graphs)
    h = lg.LeidenBatch(vseg, off, idx, w, tuning=SHAPES[blocks])
    try:
        memb, q, _ = h.run(mode=lg.LEIDEN_DETERMINISTIC)
        memb = memb.cpu().numpy()
    finally:
        h.close()
    for k, g in enumerate(graphs):
        ref = oracle.leiden(g, mode=oracle.SYNC)
        assert np.array_equal(memb[vseg[k]:vseg[k + 1]], ref.membership), k
        assert abs(q[k] - ref.modularity) <= 1e-9 * max(1.0, abs(ref.modularity))
