"""FP64 rows on either side of the degree from which the class sums are a
thread block's (257) instead of a warp's, against the oracle, with few and
many classes of neighbour degrees; also with the hub line below it and next
to it (the bin of the split rows empty, and one degree wide).  Tolerances are
those of the parity tests; FP32C takes one kernel for both sides."""
import numpy as np
import pytest

import synth
from test_gpu_device_check import _alloc, _dev, _host, ctx  # noqa: F401
from test_gpu_parity import alg1_ref, assert_parity

pytestmark = pytest.mark.gpu


def _graph():
    """A node of every degree 255..258, 512 and 513, once with 2 and once with up to 90 classes of neighbour degrees."""
    edges, n = [], 0
    for d in (255, 256, 257, 258, 512, 513):
        for classes in (2, 90):
            leaves = np.arange(d) % classes
            nb = n + 1 + np.arange(d)
            first = n + 1 + d
            edges += [np.stack([np.full(d, n), nb], 1),
                      np.stack([np.repeat(nb, leaves), first + np.arange(leaves.sum())], 1)]
            n = first + int(leaves.sum())
    return synth.relabel(synth.from_edges(n, np.concatenate(edges)), np.random.default_rng(2).permutation(n))


@pytest.mark.parametrize("precision", ["fp64", "fp32c"])
@pytest.mark.parametrize("hub_min", [33, 257, 258, 513])
def test_rows_at_the_split(ctx, hub_min, precision):  # noqa: F811
    import paper_2306_00606_gb300 as ef
    g = _graph()
    res = _alloc(g.n)
    ef.ef_set_tuning(ctx.handle, dict(row_thread_max=32, hub_min=hub_min, tri_variant=0, grid_per_sm=64, layout=0))
    try:
        ef.ef_compute_ex(ctx.handle, _dev(g.row_ptr), _dev(g.col_idx), precision=precision, **res)
    finally:
        ef.ef_set_tuning(ctx.handle, None)
    assert_parity(_host(res), alg1_ref(g), precision)
    rows = np.flatnonzero(g.degrees >= 255).astype(np.int32)
    got = _alloc(len(rows))
    ef.ef_compute_nodes(ctx.handle, _dev(g.row_ptr), _dev(g.col_idx), _dev(rows), precision=precision,
                        ef=got["ef"], s=got["s"])
    np.testing.assert_array_equal(_host(got)["s"], alg1_ref(g)["S"][rows])
    np.testing.assert_allclose(_host(got)["ef"], alg1_ref(g)["EF"][rows], rtol=1e-9 if precision == "fp64" else 0,
                               atol=1e-12 if precision == "fp64" else 2e-5)
