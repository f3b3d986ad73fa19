"""What ef_get_stats says of profiled calls: the kernels that a call launches,
against the launches that the CUDA profiler records, for every path a call can
take and every way it is decided; the pass that the fused kernel of graphs
without long rows is booked under; what a replayed graph does with other output
buffers; and what the autotuner may learn from such a graph."""
import json

import numpy as np
import pytest

import synth
from test_gpu_device_check import _alloc, _dev, ctx  # noqa: F401

pytestmark = pytest.mark.gpu

MODES = {"host": {}, "device": {"device_check": True}, "trusted": {"trust_input": True}}
GRAPHS = {
    "short": lambda: synth.watts_strogatz(3000, 8, 0.1, 1),
    "no_long_lists": lambda: synth.barabasi_albert(3000, 5, 2),
    "long_lists": lambda: synth.disjoint_union([synth.complete(90), synth.powerlaw_cm(4000, 2.1, 2, 700, 3)]),
}


def _recorded(fn, tmp_path, cat=("kernel",)):
    """Names of the kernels launched by fn, or of records of other kinds (None when no kernel can be recorded here)."""
    import torch
    from torch.profiler import ProfilerActivity, profile

    def record(f, cat=("kernel",)):
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            f()
            torch.cuda.synchronize()
        p.export_chrome_trace(str(tmp_path / "trace.json"))
        return [e["name"] for e in json.load(open(tmp_path / "trace.json"))["traceEvents"] if e.get("cat") in cat]

    x = torch.ones(8, device="cuda")
    for _ in range(3):   # the first session may record nothing
        if record(lambda: x.add_(1)):
            return record(fn, cat)
    return None


@pytest.mark.parametrize("wedge_mode", [0, 1])
@pytest.mark.parametrize("mode", list(MODES))
@pytest.mark.parametrize("name", list(GRAPHS))
def test_kernels_of_a_call(ctx, tmp_path, name, mode, wedge_mode):  # noqa: F811
    import paper_2306_00606_gb300 as ef
    g = GRAPHS[name]()
    rp, ci, res = _dev(g.row_ptr), _dev(g.col_idx), _alloc(g.n)

    def call():
        ef.ef_compute_ex(ctx.handle, rp, ci, precision="fp32c", profile=True, wedge_mode=wedge_mode, **MODES[mode], **res)

    for layout in (1, 2):
        before = ef.ef_get_tuning(ctx.handle)
        ef.ef_set_tuning(ctx.handle, dict(before, layout=layout))
        try:
            call()
            ctx.stats(reset=True)
            names = _recorded(call, tmp_path)
            if names is None:
                pytest.skip("no kernel records on this machine")
            assert len(names) == ctx.stats(reset=True)["kernels"], sorted(names)
        finally:
            ef.ef_set_tuning(ctx.handle, before)


@pytest.mark.parametrize("mode", list(MODES))
def test_fused_kernel_is_booked_as_small_wedges(ctx, mode):  # noqa: F811
    """2M nodes: about 0.4 ms of fused kernel beside an f table and launches of 0.1 ms at most."""
    import paper_2306_00606_gb300 as ef
    g = synth.watts_strogatz(2_000_000, 8, 0.1, 1)
    rp, ci, res = _dev(g.row_ptr), _dev(g.col_idx), _alloc(g.n)
    for _ in range(3):
        ctx.stats(reset=True)
        ef.ef_compute_ex(ctx.handle, rp, ci, profile=True, **MODES[mode], **res)
    st = ctx.stats(reset=True)
    assert st["wedge_small_ms"] > 2 * (st["orient_ms"] + st["tri_pairs_ms"] + st["wedge_big_ms"]), st


@pytest.mark.parametrize("mode", list(MODES))
@pytest.mark.parametrize("name", list(GRAPHS))
def test_replay_with_other_outputs(ctx, tmp_path, name, mode):  # noqa: F811
    """Calls with one captured graph and changing output buffers (others, fewer, none, the first again): right
    results, nothing written to the buffers of another call, and no second instantiation."""
    import paper_2306_00606_gb300 as ef
    g = GRAPHS[name]()
    rp, ci = _dev(g.row_ptr), _dev(g.col_idx)
    want = {k: v.clone() for k, v in _alloc(g.n).items()}
    ef.ef_compute_ex(ctx.handle, rp, ci, precision="fp64", **want)
    sets = [_alloc(g.n), _alloc(g.n), {"ef": _alloc(g.n)["ef"]}, {}, {"triangles": _alloc(g.n)["triangles"]}]
    ctx.stats(reset=True)

    def call(res):
        ef.ef_compute_ex(ctx.handle, rp, ci, precision="fp64", graph=True, **MODES[mode], **res)

    call(sets[0])   # captured
    for i in (1, 2, 3, 4, 0, 1):
        for res in sets:
            for v in res.values():
                v.fill_(7)
        names = _recorded(lambda: call(sets[i]), tmp_path, ("cuda_runtime", "cuda_driver"))
        if names is not None:
            assert any("GraphLaunch" in x for x in names) and not any("Instantiate" in x for x in names), names
        for j, res in enumerate(sets):
            for k, v in res.items():
                if j == i and k in ("ef", "t"):   # sums by atomics: equal up to their order
                    np.testing.assert_allclose(v.cpu().numpy(), want[k].cpu().numpy(), rtol=1e-12)
                elif j == i:
                    assert (v == want[k]).all(), k
                else:
                    assert (v == 7).all(), (i, j, k)
    assert ctx.stats(reset=True)["graph_replays"] == 0
    call(sets[1])
    assert ctx.stats(reset=True)["graph_replays"] == 1


@pytest.mark.parametrize("kw", [{}, {"trust_input": True}])
def test_autotune_on_short_rows_keeps_what_it_cannot_measure(ctx, kw):  # noqa: F811
    """No row above degree 32: row_thread_max, hub_min, tri_variant and layout reach no kernel that such a graph runs."""
    import torch
    import paper_2306_00606_gb300 as ef
    g = synth.watts_strogatz(4000, 8, 0.1, 5)
    rp, ci = torch.from_numpy(g.row_ptr).cuda(), torch.from_numpy(g.col_idx).cuda()
    start = dict(row_thread_max=13, hub_min=200, tri_variant=1, grid_per_sm=40, layout=2)
    ef.ef_set_tuning(ctx.handle, start)
    try:
        best = ef.ef_autotune(ctx.handle, rp, ci, precision="fp32c", reps=2, **kw)
        assert {k: v for k, v in best.items() if k != "grid_per_sm"} == \
            {k: v for k, v in start.items() if k != "grid_per_sm"}
        assert ef.ef_get_tuning(ctx.handle) == best
    finally:
        ef.ef_set_tuning(ctx.handle, None)
