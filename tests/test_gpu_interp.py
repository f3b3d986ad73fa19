"""FP64 class sums of the hub kernel by interpolation, against the oracle.

Hubs whose neighbour degrees put more and fewer classes than the threshold
(32) into an octave of y = a + D_u - 3, classes of large degree (a class each,
duplicates), octaves below 512 (integer-rounded nodes; hub_min = 33), more
classes than shared memory holds, and octaves whose last node would leave the
f table.  T within 1e-11 relative: a chunk of 32 terms is within 3.6e-12 of
its sum, and interpolation in 16 nodes magnifies the nodes' errors by at most
(2 / pi) ln 16 + 1 < 2.8."""
import numpy as np
import pytest

import oracle
import synth
from test_gpu_device_check import _dev, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


def _hub_graph(neighbour_degrees, hubs, seed):
    """`hubs` hubs joined to the same nodes, neighbour i raised to about neighbour_degrees[i] by leaves of its own."""
    k = len(neighbour_degrees)
    nb = np.arange(hubs, hubs + k)
    e = [np.stack([np.repeat(np.arange(hubs), k), np.tile(nb, hubs)], 1)]
    extra = np.maximum(np.asarray(neighbour_degrees) - hubs, 0)
    first = hubs + k
    e.append(np.stack([np.repeat(nb, extra), first + np.arange(extra.sum())], 1))
    n = first + int(extra.sum())
    g = synth.from_edges(n, np.concatenate(e))
    return synth.relabel(g, np.random.default_rng(seed).permutation(n))


CASES = {
    # D_u = 600: 31, 32 and 33 classes in the octave [1024, 2048) of y, many below
    "threshold_31": (list(range(2, 427)) + list(range(600, 600 + 31)) + [5] * (175 - 31), 1),
    "threshold_32": (list(range(2, 427)) + list(range(600, 600 + 32)) + [5] * (175 - 32), 1),
    "threshold_33": (list(range(2, 427)) + list(range(600, 600 + 33)) + [5] * (175 - 33), 1),
    # one degree only; and large degrees with duplicates (classes of one neighbour each)
    "one_class": ([7] * 700, 2),
    "large": (list(range(3, 520)) + [2050 + 40 * i for i in range(40)] + [3000] * 60, 1),
    # the hub itself has the largest degree: y reaches twice it, beyond the table's last octave
    "top_octave": (list(range(1, 1000)) + list(range(400, 1000)), 1),
}


@pytest.mark.parametrize("hub_min", [513, 129, 33])
@pytest.mark.parametrize("name", list(CASES))
def test_interpolated_class_sums(ctx, name, hub_min):  # noqa: F811
    import torch

    import paper_2306_00606_gb300 as ef
    g = _hub_graph(*CASES[name], seed=3)
    ref = oracle.vertex(g)
    ef.ef_set_tuning(ctx.handle, dict(row_thread_max=32, hub_min=hub_min, tri_variant=0, grid_per_sm=64, layout=0))
    try:
        out = ctx.compute(_dev(g.row_ptr), _dev(g.col_idx), outputs=("ef", "s", "t"))
    finally:
        ef.ef_set_tuning(ctx.handle, None)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(out["s"].cpu().numpy(), ref["S"])
    np.testing.assert_allclose(out["t"].cpu().numpy(), ref["T"], rtol=1e-11, atol=1e-12)
    np.testing.assert_allclose(out["ef"].cpu().numpy(), ref["EF"], rtol=1e-9, atol=1e-12)


def test_more_classes_than_shared_memory(ctx):  # noqa: F811
    """A hub joined to every node of a power-law graph whose degrees above 2048 are many: over 3072 classes."""
    import torch
    g0 = synth.powerlaw_cm(6000, 1.3, 900, 5900, 5)
    src = np.repeat(np.arange(g0.n), np.diff(g0.row_ptr))
    e = np.stack([src, g0.col_idx], 1)
    e = np.concatenate([e[e[:, 0] < e[:, 1]], np.stack([np.full(g0.n, g0.n), np.arange(g0.n)], 1)])
    g = synth.from_edges(g0.n + 1, e)
    d = g.degrees
    assert len(np.unique(d[d < 2048])) + (d >= 2048).sum() > 3072 + 1
    nodes = np.concatenate([[g0.n], np.argsort(-d)[:5], np.arange(10)])
    out = ctx.compute(_dev(g.row_ptr), _dev(g.col_idx), outputs=("s", "t"))
    torch.cuda.synchronize()
    ref = oracle.vertex(g, nodes.astype(np.int32))
    np.testing.assert_array_equal(out["s"].cpu().numpy()[nodes], ref["S"])
    np.testing.assert_allclose(out["t"].cpu().numpy()[nodes], ref["T"], rtol=1e-11, atol=1e-12)
