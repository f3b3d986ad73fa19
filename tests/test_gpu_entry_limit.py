"""The row pass on a graph two entries below the limit of 2^31 whose last rows
are the longest: indices one step past the end of the last row do not fit 31
bits.  The hubs are above EF_MAX_DEGREE, so the call ends after the row pass, in
an error that names their degree; nothing else of it runs.  Needs about 90 GB."""
import pytest

pytestmark = pytest.mark.gpu

HUBS = 63
LEAVES = ((1 << 30) - 1) // HUBS   # complete bipartite: exactly 2^31 - 2 entries


def test_last_row_ends_at_the_limit():
    import torch
    import paper_2306_00606_gb300 as ef
    if torch.cuda.mem_get_info()[0] < 120 << 30:
        pytest.skip("needs 120 GB of free device memory")
    n, m = LEAVES + HUBS, 2 * HUBS * LEAVES
    assert m == (1 << 31) - 2
    deg = torch.full((n,), HUBS, dtype=torch.int64, device="cuda")
    deg[LEAVES:] = LEAVES
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(deg, 0, out=rp[1:])
    assert int(rp[-1]) == m
    rp = rp.to(torch.int32)
    ci = torch.empty(m, dtype=torch.int32, device="cuda")
    half = HUBS * LEAVES
    ci[:half].view(LEAVES, HUBS).copy_(torch.arange(LEAVES, n, dtype=torch.int32, device="cuda").expand(LEAVES, HUBS))
    ci[half:].view(HUBS, LEAVES).copy_(torch.arange(LEAVES, dtype=torch.int32, device="cuda").expand(HUBS, LEAVES))
    out = torch.empty(n, dtype=torch.float64, device="cuda")
    with ef.Context(0) as ctx:
        for kw in ({}, {"device_check": True}):
            with pytest.raises(ef.EfError) as e:
                ef.ef_compute_ex(ctx.handle, rp, ci, ef=out, **kw)
            assert e.value.code == ef.EF_ERR_UNSUPPORTED and "maximum degree" in ef.ef_last_error(ctx.handle)
    del ci, rp, deg, out
    torch.cuda.empty_cache()
