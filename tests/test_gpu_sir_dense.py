"""Pull steps of the SIR simulation (dense frontiers) against the oracle, at
the edges of their lane geometry: 1, 2, 3, 9 and 32 words of simulations per
node (4, 2 and 1 nodes per warp step), rows longer than the entries loaded
ahead, rows with a warp (33 .. 128) and with a CTA each, isolated index cases,
and runs that go from push to pull and back.  Everything is exact."""
import numpy as np
import pytest

import synth
from oracle import sir
from test_gpu_device_check import _dev, ctx  # noqa: F401

pytestmark = pytest.mark.gpu

GRAPHS = {
    "ba": lambda: synth.barabasi_albert(1500, 5, 3),
    "rows": lambda: synth.disjoint_union([synth.star(40), synth.star(300), synth.complete(34), synth.path(37),
                                          synth.from_edges(3, []), synth.watts_strogatz(200, 12, 0.2, 1)]),
}


@pytest.mark.parametrize("sims", [1, 33, 70, 260, 1000])
@pytest.mark.parametrize("name", list(GRAPHS))
def test_pull_steps_match_oracle(ctx, name, sims):  # noqa: F811
    import torch
    g = GRAPHS[name]()
    rng = np.random.default_rng(sims)
    idx = rng.integers(0, g.n, sims).astype(np.int32)
    idx[: sims // 4] = int(np.argmax(g.degrees))      # several simulations from one node: dense words
    ref = sir.simulate(g, idx, 0.3, 1 / 3, seed=11)
    out = ctx.sir(_dev(g.row_ptr), _dev(g.col_idx), _dev(idx), beta=0.3, gamma=1 / 3, seed=11,
                  outputs=("final_size", "length", "peak_infected", "peak_step", "parent"))
    torch.cuda.synchronize()
    for k in ("final_size", "length", "peak_infected", "peak_step", "parent"):
        np.testing.assert_array_equal(out[k].cpu().numpy(), ref[k], err_msg=k)
