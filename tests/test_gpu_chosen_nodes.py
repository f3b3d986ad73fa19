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
