"""The fused kernel of graphs without long rows takes 2, 8 or 32 nodes per
warp step by the number of nodes.  Copies of one graph of mixed short rows
(full rows of 32, isolated nodes, stars) at sizes of each form, just below and
above its first size; the copies' length shares no factor with a step, so that
every row is met at every place of a step.  Each copy against the oracle's
results of the one graph."""
import numpy as np
import pytest

import synth
from test_gpu_device_check import _alloc, _dev, _host, ctx  # noqa: F401
from test_gpu_parity import alg1_ref, assert_parity
from test_gpu_short_rows import _bins_graph

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32c"])
@pytest.mark.parametrize("per_sm,extra", [(256, -1), (256, 1), (1024, -1), (1024, 33)])
def test_steps_of_2_8_and_32_nodes(ctx, per_sm, extra, precision):  # noqa: F811
    import torch
    import paper_2306_00606_gb300 as ef
    g = _bins_graph()
    if g.n % 2 == 0:
        g = synth.disjoint_union([g, synth.from_edges(1, [])])
    assert g.degrees.max() == 32 and (g.degrees == 0).any()
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + extra
    copies, rest = divmod(n, g.n)
    rp = np.concatenate([g.row_ptr[:-1].astype(np.int64) + i * g.nnz for i in range(copies)]
                        + [np.full(rest + 1, copies * g.nnz, np.int64)]).astype(np.int32)
    ci = np.concatenate([g.col_idx.astype(np.int64) + i * g.n for i in range(copies)]).astype(np.int32)
    ref = alg1_ref(g)
    lone = int(np.flatnonzero(g.degrees == 0)[0])
    ref = {k: np.concatenate([np.tile(v, copies), np.full(rest, v[lone], v.dtype)]) for k, v in ref.items()
           if k in ("N", "S", "T", "EF", "flag", "tri")}
    res = _alloc(n)
    ef.ef_compute_ex(ctx.handle, _dev(rp), _dev(ci), precision=precision, **res)
    assert_parity(_host(res), ref, precision)
