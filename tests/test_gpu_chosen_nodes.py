"""Exact EF of chosen nodes with and without the filter that keeps credits from
nodes off the list (used from 2^21 nodes on; the same graph padded with
isolated nodes takes it), against the oracle: every bin of middle nodes, rows
above the marking kernel's block line (512), lists with a node twice, ids at
both ends, triangles by pairs and by streaming.  Tolerances are those of the
parity tests."""
import numpy as np
import pytest

import synth
from test_gpu_device_check import _alloc, _dev, _host, ctx  # noqa: F401
from test_gpu_parity import alg1_ref, assert_parity

pytestmark = pytest.mark.gpu

FILTER_FROM = 1 << 21


def _graph():
    g = synth.disjoint_union([synth.powerlaw_cm(6000, 2.1, 2, 900, 5), synth.complete(40), synth.star(700),
                              synth.complete(300), synth.watts_strogatz(500, 6, 0.2, 6), synth.path(2)])
    return synth.relabel(g, np.random.default_rng(7).permutation(g.n))


@pytest.mark.parametrize("precision", ["fp64", "fp32c"])
@pytest.mark.parametrize("pad", [0, FILTER_FROM])
@pytest.mark.parametrize("share", [1.0, 0.02])
def test_chosen_nodes_match_oracle(ctx, share, pad, precision):  # noqa: F811
    import paper_2306_00606_gb300 as ef
    g = _graph()
    rng = np.random.default_rng(8)
    rows = np.flatnonzero(rng.random(g.n) < share)
    rows = np.concatenate([rows, [0, g.n - 1, int(np.argmax(g.degrees)), rows[0]]]).astype(np.int32)
    rp = np.concatenate([g.row_ptr, np.full(max(pad - g.n, 0), g.row_ptr[-1])]).astype(np.int32)
    got = _alloc(len(rows))
    ef.ef_compute_nodes(ctx.handle, _dev(rp), _dev(g.col_idx), _dev(rows), precision=precision, **got)
    ref = {k: v[rows] for k, v in alg1_ref(g).items()}
    assert_parity(_host(got), ref, precision)


@pytest.mark.parametrize("past", [0, 1])
def test_listed_share_at_the_filters_line(ctx, past):  # noqa: F811
    """The filter is used up to a listed share of n / 25e6: lists (with repeats) on either side, fp64 and fp32c alike."""
    import paper_2306_00606_gb300 as ef
    g, n = _graph(), FILTER_FROM
    rows = np.resize(np.random.default_rng(9).permutation(g.n), int(n * n / 25e6) + past).astype(np.int32)
    rp = np.concatenate([g.row_ptr, np.full(n - g.n, g.row_ptr[-1])]).astype(np.int32)
    ref = {k: v[rows] for k, v in alg1_ref(g).items()}
    for precision in ("fp64", "fp32c"):
        got = _alloc(len(rows))
        ef.ef_compute_nodes(ctx.handle, _dev(rp), _dev(g.col_idx), _dev(rows), precision=precision, **got)
        assert_parity(_host(got), ref, precision)


@pytest.mark.parametrize("precision", ["fp64", "fp32c"])
@pytest.mark.parametrize("k", [1, 911, 913, 7297, 58369, 120001])
def test_nodes_by_warps_and_by_blocks(ctx, k, precision):  # noqa: F811
    """List lengths around one node per block and around one and two nodes per warp step, over nodes of 0, 1, 2, 31,
    32 and 33 neighbours and more, triangles by pairs and by streaming; ids outside the graph are refused in each."""
    import paper_2306_00606_gb300 as ef
    pairs = synth.from_edges(3000, [(0, j) for j in range(1, 2049)] + [(2100, j) for j in range(2101, 3000)] + [(1, 2)])
    g = synth.disjoint_union([synth.powerlaw_cm(4000, 2.2, 2, 500, 5), synth.complete(32), synth.complete(33),
                              synth.complete(34), synth.watts_strogatz(600, 6, 0.2, 6), synth.star(30), synth.path(2),
                              synth.from_edges(2, []), pairs])
    ref = alg1_ref(g)
    rows = np.resize(np.random.default_rng(k).permutation(g.n), k).astype(np.int32)
    rp, ci, got = _dev(g.row_ptr), _dev(g.col_idx), _alloc(k)
    ef.ef_compute_nodes(ctx.handle, rp, ci, _dev(rows), precision=precision, **got)
    assert_parity(_host(got), {key: v[rows] for key, v in ref.items()}, precision)
    for bad in (-1, g.n):
        with pytest.raises(ef.EfError):
            ef.ef_compute_nodes(ctx.handle, rp, ci, _dev(np.append(rows[:-1], bad).astype(np.int32)), **got)


def test_list_much_longer_than_the_graph(ctx):  # noqa: F811
    """From position 2 n on also nodes of more than 32 neighbours go by warps."""
    import paper_2306_00606_gb300 as ef
    g = synth.disjoint_union([synth.complete(34), synth.star(40), synth.path(3)])
    rows = np.tile(np.arange(g.n, dtype=np.int32), 7)
    got = _alloc(len(rows))
    ef.ef_compute_nodes(ctx.handle, _dev(g.row_ptr), _dev(g.col_idx), _dev(rows), **got)
    assert_parity(_host(got), {key: v[rows] for key, v in alg1_ref(g).items()}, "fp64")
