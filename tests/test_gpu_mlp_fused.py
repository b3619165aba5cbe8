"""The warm-start network's whole-network kernels at the edges of their tiles:
widths that end inside and on a 16-feature step and a 128-feature block (one
and two accumulator tiles), batches of one row, around the 16-row steps and
over several rounds of tiles, two to sixteen layers (the deepest train layer
by layer), 1 and 16 inputs and outputs; and a network too wide for them.

Against oracle/mlp.py in bfloat16 mode, which rounds what the kernels round.
Tolerances: each hidden layer rounds its activations to bfloat16 (2^-9), and a
value near a rounding boundary may fall on the other side of it because the
FP32 sums differ in their last bits; the four-layer networks of
test_gpu_mlp.py are held to 2e-3 (forward) and 1e-2 (gradient), and each layer
adds as much again: those bounds times n_layers / 4 (at least 1).
"""
import numpy as np
import pytest

import lbm_inputs as I
from oracle import mlp as M

pytestmark = pytest.mark.gpu

SHAPES = [  # n_in, width, layers, n_out, rows
    (7, 256, 4, 3, 1), (7, 256, 4, 3, 15), (7, 256, 4, 3, 17), (7, 256, 4, 3, 2433),
    (7, 256, 4, 3, 10000), (1, 16, 2, 1, 33), (16, 17, 3, 16, 48), (8, 128, 3, 9, 4864),
    (7, 129, 3, 3, 300), (9, 240, 5, 4, 97), (7, 256, 2, 16, 640), (7, 256, 16, 3, 200),
    (7, 320, 3, 3, 150),
]


def _rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / max(np.linalg.norm(b), 1e-300))


@pytest.mark.parametrize("shape", SHAPES)
def test_forward_and_gradient_match_the_oracle(shape):
    import torch
    from paper_2108_08783_gb300 import MLP
    n_in, width, n_layers, n_out, n = shape
    net = MLP(n_in, width, n_layers, n_out, max_batch=n)
    theta = I.mlp_init(3, n_in, width, n_layers, n_out, bias_scale=0.1)
    net.set_params(theta)
    x, t = I.mlp_batch(4, n, n_in, n_out, scale=0.5)
    xd, td = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    sizes = M.layer_sizes(n_in, width, n_layers, n_out)
    grow = max(1.0, n_layers / 4)
    # rows beyond the batch stay as they are
    y = torch.full((n + 4, n_out), 7.0, device="cuda")
    import ctypes as C
    net._check(net._lib.lbm_mlp_forward(net.h, C.c_void_p(xd.data_ptr()), n,
                                        C.c_void_p(y.data_ptr())))
    net.sync()
    y = y.cpu().numpy()
    assert np.all(y[n:] == 7.0)
    y_ref, _ = M.forward(theta, sizes, x, bf16=True)
    assert _rel(y[:n], y_ref) < 2e-3 * grow
    loss, g = net.loss_grad(xd, td)
    net.sync()
    E, g_ref = M.loss_grad(theta, sizes, x, t, bf16=True)
    assert abs(loss - E) <= 1e-3 * grow * E
    assert _rel(g, g_ref) < 1e-2 * grow
    # a second pass over the same batch gives the same gradient
    loss2, g2 = net.loss_grad(xd, td)
    if width <= 256 and n_layers <= 4:  # the whole-network kernels add in a fixed order
        assert loss2 == loss and np.array_equal(g, g2)


def test_more_rows_than_the_batch_and_training_after_it():
    """A forward pass of any number of rows, and the weights a step leaves are
    the ones the next forward pass uses."""
    import torch
    from paper_2108_08783_gb300 import MLP
    theta = I.mlp_init(5, 7, 256, 4, 3)
    x, t = I.mlp_batch(6, 50000, 7, 3)
    xd, td = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    net = MLP(7, 256, 4, 3, max_batch=512)
    net.set_params(theta)
    net.train_step(xd[:512], td[:512], lr=1e-2)
    y = net.forward(xd)
    net.sync()
    other = MLP(7, 256, 4, 3, max_batch=512)
    other.set_params(net.params())
    parts = [other.forward(xd[k:k + 777]) for k in range(0, 50000, 777)]
    other.sync()
    assert torch.equal(y, torch.cat(parts))
