"""Out-list hash tables with two slots per entry (no node has more than 24
out-neighbours) and with three (some node has), filled by one thread (rows up
to degree 32) and by the lanes of a warp: lists of every length from the first
that has a table (6) to 24, 33 and beyond, dense parts in which most probes find
their key and sparse ones in which most do not, both list layouts, both ways of
clearing.  Triangle counts are exact, the rest within the parity tests'
tolerances."""
import numpy as np
import pytest

import synth
from test_gpu_device_check import _alloc, _dev, _host, ctx  # noqa: F401
from test_gpu_parity import alg1_ref, assert_parity

pytestmark = pytest.mark.gpu


def _graph(longest):
    """Complete graphs K_6 .. K_longest (out-lists of 0 .. longest - 1 entries) beside random parts, shuffled ids."""
    parts = [synth.complete(k) for k in range(6, longest + 1)]
    parts += [synth.erdos_renyi(700, 0.02, 3), synth.barabasi_albert(900, 12, 4), synth.complete_bipartite(20, 40)]
    g = synth.disjoint_union(parts)
    return synth.relabel(g, np.random.default_rng(longest).permutation(g.n))


@pytest.mark.parametrize("mode", [{}, {"device_check": True}, {"trust_input": True, "graph": True}])
@pytest.mark.parametrize("layout", [1, 2])
@pytest.mark.parametrize("rows", [8, 32])
@pytest.mark.parametrize("longest", [24, 25, 26, 33, 34, 60])
def test_tables_of_every_length(ctx, longest, rows, layout, mode):  # noqa: F811
    import paper_2306_00606_gb300 as ef
    g = _graph(longest)
    assert g.degrees.max() > 32
    before, got = ef.ef_get_tuning(ctx.handle), _alloc(g.n)
    ef.ef_set_tuning(ctx.handle, dict(before, layout=layout, row_thread_max=rows))
    try:
        ef.ef_compute_ex(ctx.handle, _dev(g.row_ptr), _dev(g.col_idx), precision="fp64", **mode, **got)
    finally:
        ef.ef_set_tuning(ctx.handle, before)
    assert_parity(_host(got), alg1_ref(g), "fp64")
