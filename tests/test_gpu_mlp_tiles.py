"""Training batches of several tiles per CTA of the whole-network kernels.

The barriers of forward and back-propagation are waited on by phase parity, so
each has to be seen before its next phase can complete, also where a tile's
last error is followed by the next tile's inputs.  152 CTAs of at most 64 rows:
30,011 rows are three to four tiles each, the last one ragged; width 100 ends
inside a warp's 32 features (112 with its padding).

Against oracle/mlp.py in bfloat16 mode, with the bounds of the whole-network
kernels' other tests: 1e-3 for the loss and 1e-2 for the gradient (a value near
a bfloat16 rounding boundary may fall on the other side); the kernels add in a
fixed order, so a second pass gives the same bits.
"""
import numpy as np
import pytest

import lbm_inputs as I
from oracle import mlp as M

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 16, 2, 1, 30011), (16, 100, 3, 16, 20001),
                                   (7, 256, 4, 3, 19999)])
def test_gradient_over_several_tiles_per_cta(shape):
    import torch
    from paper_2108_08783_gb300 import MLP
    n_in, width, n_layers, n_out, n = shape
    net = MLP(n_in, width, n_layers, n_out, max_batch=n)
    theta = I.mlp_init(3, n_in, width, n_layers, n_out, bias_scale=0.1)
    net.set_params(theta)
    x, t = I.mlp_batch(4, n, n_in, n_out, scale=0.5)
    xd, td = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    sizes = M.layer_sizes(n_in, width, n_layers, n_out)
    loss, g = net.loss_grad(xd, td)
    net.sync()
    E, g_ref = M.loss_grad(theta, sizes, x, t, bf16=True)
    assert abs(loss - E) <= 1e-3 * E
    assert np.linalg.norm(np.asarray(g, np.float64) - g_ref) < 1e-2 * np.linalg.norm(g_ref)
    for _ in range(20):
        loss2, g2 = net.loss_grad(xd, td)
        net.sync()
        assert loss2 == loss and np.array_equal(g, g2)


@pytest.mark.parametrize("width", [48, 100, 208, 272])
def test_widths_that_end_inside_a_warp(width):
    """Half of a warp's lanes leave the epilogue's stores out before the next
    collective load from tensor memory (272: the layer-by-layer kernel, whose
    rows beyond the batch do)."""
    import torch
    from paper_2108_08783_gb300 import MLP
    n = 177
    net = MLP(5, width, 3, 9, max_batch=n)
    theta = I.mlp_init(3, 5, width, 3, 9, bias_scale=0.1)
    net.set_params(theta)
    x, t = I.mlp_batch(4, n, 5, 9, scale=0.5)
    sizes = M.layer_sizes(5, width, 3, 9)
    xd, td = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    y = net.forward(xd)
    loss, g = net.loss_grad(xd, td)
    net.sync()
    y_ref, _ = M.forward(theta, sizes, x, bf16=True)
    E, g_ref = M.loss_grad(theta, sizes, x, t, bf16=True)
    assert np.linalg.norm(y.cpu().numpy() - y_ref) < 2e-3 * np.linalg.norm(y_ref)
    assert abs(loss - E) <= 1e-3 * E
    assert np.linalg.norm(np.asarray(g, np.float64) - g_ref) < 1e-2 * np.linalg.norm(g_ref)
