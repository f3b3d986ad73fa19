"""The direction of SIR steps (push, pull) against the oracle.  The oracle's own
draws say which nodes are infected at each step, and with them whether a step
pulls: once the infected nodes' rows hold more than half of all entries, or a
third from eight words (more than 224 simulations) on.
Every case is shown to take the directions it is there for.  Sizes at the edges
of a pull step's share: one group of nodes per warp (small graphs) up to the
full eight, with a last share that is not full.  Everything is exact."""
import numpy as np
import pytest

import synth
from oracle import sir
from test_gpu_device_check import _dev, ctx  # noqa: F401

OUTS = ("final_size", "length", "peak_infected", "peak_step", "parent")


def _dense(sims):
    """A step pulls when this many times the frontier's entries exceed all entries."""
    return 3 if sims > 224 else 2


# graph, simulations, R0, and whether a push step follows a pull step
CASES = {
    "ba_1_sim": (lambda: synth.barabasi_albert(1500, 5, 3), 1, 9.0, True),
    "ba_33_sims": (lambda: synth.barabasi_albert(1500, 5, 3), 33, 3.0, True),
    "hubs_70_sims": (lambda: synth.powerlaw_cm(3000, 2.1, 3, 800, 5), 70, 2.0, True),
    "er_7_words": (lambda: synth.erdos_renyi(4865, 0.002, 6), 224, 2.0, True),
    "er_8_words": (lambda: synth.erdos_renyi(4865, 0.002, 6), 225, 2.0, True),
    "er_9_words": (lambda: synth.erdos_renyi(4865, 0.002, 6), 260, 1.5, True),
    "share_3_of_1_word": (lambda: synth.barabasi_albert(45001, 4, 7), 20, 3.0, True),
    "share_3_of_5_words": (lambda: synth.barabasi_albert(9999, 5, 8), 130, 2.0, True),
    "share_8": (lambda: synth.erdos_renyi(45003, 0.0002, 9), 100, 2.0, True),
    "all_words_first_step_pulls": (lambda: synth.complete(70), 1000, 3.0, False),
}


def _oracle(name):
    """Graph, call arguments, oracle outputs, and per step whether it pulls."""
    make, sims, r0, _ = CASES[name]
    g = make()
    rng = np.random.default_rng(sims)
    idx = rng.integers(0, g.n, sims).astype(np.int32)
    args = dict(beta=min(1.0, r0 / (3 * g.nnz / g.n)), gamma=1 / 3, seed=11)
    frontiers, draw = [], sir.philox4x32_10

    def record(c0, c1, c2, c3, key):
        if np.size(c3) and int(np.ravel(c3)[0]) == sir.RECOVER:   # the recoveries: every infected node of the step
            frontiers.append(np.unique(c2))
        return draw(c0, c1, c2, c3, key)

    sir.philox4x32_10 = record
    try:
        ref = sir.simulate(g, idx, **args)
    finally:
        sir.philox4x32_10 = draw
    deg = np.diff(g.row_ptr).astype(np.int64)
    return g, idx, args, ref, np.array([_dense(sims) * deg[f].sum() > g.nnz for f in frontiers])


@pytest.mark.parametrize("name", list(CASES))
def test_cases_take_the_directions_they_stand_for(name):
    pulls = _oracle(name)[4]
    assert pulls.any()
    if CASES[name][3]:
        first, last = np.flatnonzero(pulls)[[0, -1]]
        assert first > 0 and last < len(pulls) - 1 and not pulls[last + 1:].any()   # push, pull, push
    else:
        assert pulls[0]


@pytest.mark.gpu
@pytest.mark.parametrize("name", list(CASES))
def test_directions_match_oracle(ctx, name):  # noqa: F811
    import torch
    g, idx, args, ref, _ = _oracle(name)
    out = ctx.sir(_dev(g.row_ptr), _dev(g.col_idx), _dev(idx), outputs=OUTS, **args)
    torch.cuda.synchronize()
    for k in OUTS:
        np.testing.assert_array_equal(out[k].cpu().numpy(), ref[k], err_msg=k)
