"""The network at row counts that leave tiles, warps and blocks partly filled,
against the CPU oracle.  Predictions of dyadic networks are exact; a gradient
over a power of two of rows is, and over other counts each element stays
within the bound of the parity tests (2^-6 of the absolute sum of its terms)."""
import numpy as np
import pytest

from netcases import dyadic_network
from oracle import surrogate as sg
from test_gpu_device_check import _dev, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


def _model(ctx, p):  # noqa: F811
    import paper_2306_00606_gb300 as ef
    m = ef.Model(ctx.handle)
    m.set(np.concatenate([sg.flatten(p), p["mean"], p["std"]]).astype(np.float32))
    return m


@pytest.mark.parametrize("rows", [1, 15, 16, 17, 31, 33, 127, 128, 129, 255, 257, "line", "line+1", "line*2+33"])
def test_forward_rows(ctx, rows):  # noqa: F811
    import torch
    line = 256 * torch.cuda.get_device_properties(0).multi_processor_count   # one 16-row tile per warp of the chip
    n = {"line": line, "line+1": line + 1, "line*2+33": 2 * line + 33}.get(rows, rows)
    p, X, _ = dyadic_network(11, n)
    out = torch.full((n + 64,), -7.0, dtype=torch.float32, device="cuda")
    _model(ctx, p).forward(_dev(X.astype(np.float32)), out[:n])
    np.testing.assert_array_equal(out[:n].cpu().numpy().astype(np.float64), sg.forward(p, X)[0])
    assert bool((out[n:] == -7.0).all())   # nothing written behind the last row


@pytest.mark.parametrize("rows", [1, 15, 16, 17, 31, 32, 33, 127, 128, 129, 255, 257, 2048])
def test_gradient_rows(ctx, rows):  # noqa: F811
    p, X, y = dyadic_network(12, rows)
    loss, grad = _model(ctx, p).grad(_dev(X.astype(np.float32)), _dev(y.astype(np.float32)))
    exact = rows & (rows - 1) == 0
    ref_loss, ref_g = sg.loss_and_grads(p, X, y, operands="fp64" if exact else "bf16")
    sums, _ = sg.grad_term_sums(p, X, y, operands="bf16")
    assert loss == ref_loss if exact else abs(loss - ref_loss) <= 2.0 ** -20 * ref_loss
    o = 0
    for k in sg.TRAINED:
        size = int(np.prod(sg.SHAPES[k]))
        a, b = grad[o:o + size].astype(np.float64), np.ravel(ref_g[k])
        tol = 0.0 if exact else 2.0 ** -6 * np.ravel(sums[k]) + 1e-12
        assert np.all(np.abs(a - b) <= tol), (k, float(np.max(np.abs(a - b))))
        o += size


def test_gradient_of_the_smallest_activations(ctx):  # noqa: F811
    """A hidden unit whose activation is positive in FP32 but rounds to 0 in BF16 is active: its bias has a gradient."""
    p, X, _ = dyadic_network(13, 32)
    p["W1"][:] = 0.0
    p["b1"] = np.resize(np.array([1e-41, 0.0, -1e-41, 0.5, 2e-45]), 64).astype(np.float32).astype(np.float64)
    y = sg.forward(p, X)[0] - 1.0
    _, grad = _model(ctx, p).grad(_dev(X.astype(np.float32)), _dev(y.astype(np.float32)))
    _, ref = sg.loss_and_grads(p, X, y)
    assert np.count_nonzero(ref["b1"][(p["b1"] > 0) & (p["b1"] < 1e-40)]) > 10
    o = 0
    for k in sg.TRAINED:
        size = int(np.prod(sg.SHAPES[k]))
        np.testing.assert_allclose(grad[o:o + size].astype(np.float64), np.ravel(ref[k]), rtol=0, atol=1e-37, err_msg=k)
        o += size
