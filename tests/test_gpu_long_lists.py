"""Pair tests of out-lists at the edges of the kernels' candidate groups: out-
degrees around 32 (the line between the two kernels), 64 and 96, lists with
and without a hash table, tables with full buckets, every pair a triangle and
almost none, for the whole graph and for shards of it.  Tolerances are those
of the parity tests (triangles, S and N are equal)."""
import numpy as np
import pytest

import synth
from test_gpu_device_check import _alloc, _dev, _host, ctx  # noqa: F401
from test_gpu_parity import alg1_ref, assert_parity
from test_gpu_shard import _close, _finalize, _shards

pytestmark = pytest.mark.gpu


def _multipartite(parts, size):
    """No edge within a part: an owner's candidates of one part miss each other's lists."""
    ids = np.arange(parts * size)
    a, b = np.triu_indices(len(ids), 1)
    keep = a // size != b // size
    return synth.from_edges(len(ids), np.stack([a[keep], b[keep]], 1))


GRAPHS = {
    # K_k: the out-degrees are 0..k-1, every pair of every out-list a triangle
    "cliques": lambda: [synth.complete(k) for k in (33, 34, 35, 65, 66, 67, 98)],
    # out-degrees about the same sizes, a quarter and a half of the pairs triangles
    "dense": lambda: [synth.erdos_renyi(260, 0.25, 1), synth.erdos_renyi(150, 0.5, 2), synth.complete(5)],
    "parts": lambda: [_multipartite(3, 33), _multipartite(2, 70), _multipartite(9, 8)],
}


def _graph(name):
    g = synth.disjoint_union(GRAPHS[name]())
    return synth.relabel(g, np.random.default_rng(4).permutation(g.n))


@pytest.mark.parametrize("precision", ["fp64", "fp32c"])
@pytest.mark.parametrize("name", list(GRAPHS))
def test_long_lists_match_oracle(ctx, name, precision):  # noqa: F811
    import paper_2306_00606_gb300 as ef
    g = _graph(name)
    ref = alg1_ref(g)
    for mode in ({}, {"device_check": True, "graph": True}):
        res = _alloc(g.n)
        ef.ef_compute_ex(ctx.handle, _dev(g.row_ptr), _dev(g.col_idx), precision=precision, **mode, **res)
        assert_parity(_host(res), ref, precision)
    _, _, tot, _, _, frac = _shards(ctx, g, 3, precision)
    got = _finalize(ctx, tot, frac, precision)
    np.testing.assert_array_equal(got["triangles"], _host(res)["triangles"])
    np.testing.assert_array_equal(got["s"], ref["S"])
    _close(got["ef"], ref["EF"], precision)


@pytest.mark.parametrize("copies", [2, 6, 25, 60, 120, 260])
def test_items_shared_among_warps(ctx, copies):  # noqa: F811
    """About 200 items a copy (a clique, a dense random part): 32, 16, 8, 4, 2 warps and one warp per item."""
    import paper_2306_00606_gb300 as ef
    one = synth.disjoint_union([synth.complete(98), synth.erdos_renyi(150, 0.5, 2)])
    ref = {k: np.tile(v, copies) for k, v in alg1_ref(one).items()}
    g = synth.disjoint_union([one] * copies)
    res = _alloc(g.n)
    ef.ef_compute_ex(ctx.handle, _dev(g.row_ptr), _dev(g.col_idx), precision="fp64", **res)
    assert_parity(_host(res), ref, "fp64")
