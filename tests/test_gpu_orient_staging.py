"""The orientation of graphs without rows above degree 32 (calls outside the
short-row path: here one shard), which stages a warp's 32 out-lists and their
tables in shared memory: 4 to 7 out-neighbours a node on average, so that the
lists of a step hold about 128, 160, 192 (the staging area) and 224 entries,
both orders of the lists.  Integers are exact, EF within the parity tests'
tolerances."""
import numpy as np
import pytest

import synth
from test_gpu_parity import EF_RTOL64, alg1_ref
from test_gpu_shard import _finalize, _shards, ctx  # noqa: F401

pytestmark = pytest.mark.gpu

GRAPHS = {f"ws_{k}": (lambda k=k: synth.watts_strogatz(3001, k, 0.05, k)) for k in (8, 10, 12, 14)}
GRAPHS["er_10"] = lambda: synth.erdos_renyi(4003, 0.0025, 3)
GRAPHS["full_rows"] = lambda: synth.disjoint_union([synth.complete(k) for k in (2, 7, 12, 13, 14, 31, 32, 33)] * 3)


@pytest.mark.parametrize("layout", [1, 2])
@pytest.mark.parametrize("name", list(GRAPHS))
def test_staged_lists_match_oracle(ctx, name, layout):  # noqa: F811
    import paper_2306_00606_gb300 as ef
    g = GRAPHS[name]()
    assert g.degrees.max() <= 32
    before = ef.ef_get_tuning(ctx.handle)
    ef.ef_set_tuning(ctx.handle, dict(before, layout=layout))
    try:
        _, _, tot, _, _, frac = _shards(ctx, g, 1)
    finally:
        ef.ef_set_tuning(ctx.handle, before)
    got, ref = _finalize(ctx, tot, frac, "fp64"), alg1_ref(g)
    for k, want in (("n_clusters", "N"), ("s", "S"), ("triangles", "tri"), ("flag", "flag")):
        np.testing.assert_array_equal(got[k], ref[want], err_msg=k)
    np.testing.assert_allclose(got["ef"], ref["EF"], rtol=EF_RTOL64, atol=1e-12)
