"""GPU test of the work counters of a profiled run (LEIDEN_FLAG_PROFILE) on
rows whose entries together pass 32 bits."""
import pytest
import torch

import paper_2312_13936_gb300 as lg

pytestmark = pytest.mark.gpu


def test_entries_beyond_32_bits():
    """17 vertices, each joined to all others and to itself 2^28 times: every
    row is the only one of its step, nobody gains by moving, and one sweep of
    each phase reads every entry of the graph once."""
    n, loops = 17, 1 << 28
    nnz = n * (loops + n - 1)
    assert nnz > 1 << 32
    if torch.cuda.mem_get_info()[0] < 24 * nnz:
        pytest.skip("needs some 110 GB of device memory")
    off = torch.arange(n + 1, dtype=torch.int64, device="cuda") * (loops + n - 1)
    idx = torch.empty(nnz, dtype=torch.int32, device="cuda")
    for v in range(n):
        row = idx[v * (loops + n - 1):(v + 1) * (loops + n - 1)]
        row.fill_(v)
        row[:n - 1] = torch.tensor([u for u in range(n) if u != v], dtype=torch.int32)
    h = lg.Leiden(off, idx)
    try:
        memb, q, st = h.run(flags=lg.FLAG_PROFILE)
        assert memb.tolist() == list(range(n))
        assert (st.move_iterations, st.refine_iterations) == (1, 1)
        prof = h.profile()
        for phase in ("move", "refine"):
            got = prof[(phase, "sweep")]
            assert got["items"] == n and got["edges"] == nnz, (phase, got)
    finally:
        h.close()
    del off, idx, row
    torch.cuda.empty_cache()
