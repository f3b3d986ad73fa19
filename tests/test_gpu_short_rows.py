"""The short-row path (no node above degree 32) against the oracle, at the
edges of its degree bins and of its warp steps, for each way a call decides
on it: by the host after the readback, and by the device (device_check,
trust_input, replayed graphs), also when a context alternates between graphs
of the two paths.  Tolerances are those of the parity tests."""
import numpy as np
import pytest

import synth
from test_gpu_device_check import OUTS, _alloc, _dev, _host, ctx  # noqa: F401
from test_gpu_parity import alg1_ref, assert_parity

pytestmark = pytest.mark.gpu

MODES = {"host": {}, "device": {"device_check": True}, "trusted": {"trust_input": True},
         "replay": {"device_check": True, "graph": True}, "host_graph": {"graph": True}}


def _bins_graph():
    """Complete graphs with degrees at every bin edge (K2..K33), isolated nodes between them, and random parts."""
    parts = []
    for k in (2, 3, 5, 6, 9, 10, 17, 18, 32, 33):
        parts += [synth.complete(k), synth.from_edges(1, [])]
    return synth.disjoint_union(parts + [synth.watts_strogatz(1000, 12, 0.2, 3), synth.erdos_renyi(700, 0.012, 4),
                                         synth.star(32), synth.path(1), synth.complete_bipartite(32, 31)])


GRAPHS = {
    "bins": _bins_graph,
    "sparse": lambda: synth.erdos_renyi(3001, 0.0007, 5),        # many isolated nodes and short components
    "two_nodes": lambda: synth.from_edges(2, [(0, 1)]),
    "no_edges": lambda: synth.from_edges(37, []),
    "degree_33": lambda: synth.disjoint_union([synth.complete(34), synth.cycle(70)]),   # first general size
    "relabelled": lambda: synth.relabel(synth.watts_strogatz(4097, 8, 0.1, 6), np.random.default_rng(1).permutation(4097)),
}


@pytest.mark.parametrize("mode", list(MODES))
@pytest.mark.parametrize("precision", ["fp64", "fp32c"])
@pytest.mark.parametrize("name", list(GRAPHS))
def test_short_rows_match_oracle(ctx, name, precision, mode):  # noqa: F811
    import paper_2306_00606_gb300 as ef
    g = GRAPHS[name]()
    big = synth.barabasi_albert(400, 5, 9)
    assert (big.degrees.max() > 32) and ((g.degrees.max() > 32) == (name == "degree_33"))
    rp, ci, res = _dev(g.row_ptr), _dev(g.col_idx), _alloc(g.n)
    rpb, cib, other = _dev(big.row_ptr), _dev(big.col_idx), _alloc(big.n)
    ref = alg1_ref(g)
    for _ in range(2):   # between calls of the other path, which uses the same scratch
        ef.ef_compute_ex(ctx.handle, rpb, cib, precision=precision, **MODES[mode], **other)
        ef.ef_compute_ex(ctx.handle, rp, ci, precision=precision, **MODES[mode], **res)
        assert_parity(_host(res), ref, precision)
    assert_parity(_host(other), alg1_ref(big), precision)


@pytest.mark.parametrize("device_check", [False, True])
def test_short_batch_graph_bounds(ctx, device_check):  # noqa: F811
    """A batch of tiny graphs (several per warp of rows): results per graph, and an entry that leaves its graph
    by one node at either end of a warp's rows is refused."""
    import paper_2306_00606_gb300 as ef
    parts = [synth.complete(k) for k in (3, 1, 4, 33, 2, 5)] * 30 + [synth.watts_strogatz(300, 6, 0.1, 1)]
    g = synth.disjoint_union(parts)
    res = _alloc(g.n)
    ef.ef_compute_batched(ctx.handle, _dev(g.row_ptr), _dev(g.col_idx), g.graph_off, device_check=device_check, **res)
    assert_parity(_host(res), alg1_ref(g), "fp64")
    for cut in (64, 100, g.n - 150):   # offsets that split an edge's ends between two graphs
        off = np.array([0, cut, g.n], np.int64)
        src = np.repeat(np.arange(g.n), np.diff(g.row_ptr))
        crosses = bool(np.any((src < cut) != (g.col_idx < cut)))
        if not crosses:
            continue
        with pytest.raises(ef.EfError) as e:
            ef.ef_compute_batched(ctx.handle, _dev(g.row_ptr), _dev(g.col_idx), off, device_check=device_check, **res)
        assert e.value.code == ef.EF_ERR_GRAPH and "edge-between-graphs" in str(e.value)
