"""The tiled convolution kernels at the edges of their tiles (32 columns, 8 or 32 rows, channel
groups of 8 and chunks of 32): odd and one-wide grids, channel counts around the groups, against
the float64 oracle.  Sums of at most 9 * 70 products per output and of B H W <= 3000 products per
weight: relative error of the vectors <= sqrt(3000) eps32 ~ 3e-6; 1e-5 (outputs) and 1e-4
(gradients, whose terms cancel) as in the tests of the whole network."""
import numpy as np
import pytest
import torch

from oracle import nn as N
from paper_2507_05222_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2507_05222_gb300 import qtt
    return qtt.Context(0)


def rel(a, b):
    a = np.asarray(a, dtype=np.float64).ravel(); b = np.asarray(b, dtype=np.float64).ravel()
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


@pytest.mark.parametrize("c_in,width,depth,B,H,W", [
    (1, 1, 1, 1, 1, 1), (1, 3, 2, 2, 3, 2), (2, 5, 3, 1, 9, 33), (4, 8, 2, 3, 8, 32), (3, 9, 3, 2, 7, 31),
    (5, 33, 2, 1, 33, 35), (4, 40, 3, 1, 17, 64), (64, 70, 2, 1, 5, 40), (4, 32, 4, 2, 32, 16), (2, 4, 2, 1, 1, 70)])
def test_forward_gradient_and_scaling(ctx, c_in, width, depth, B, H, W):
    from paper_2507_05222_gb300 import qtt
    g = inputs.rng(100 + c_in + width + H + W)
    p = []
    for co, ci in N.layer_shapes(c_in, width, depth):
        p += [g.standard_normal(co * ci * 9) * np.sqrt(2.0 / (ci * 9)), 0.1 * g.standard_normal(co)]
    p = np.concatenate(p).astype(np.float32)
    x = g.standard_normal((B, c_in, H, W)).astype(np.float32)
    y = g.standard_normal((B, 1, H, W)).astype(np.float32)
    shift, scale = g.standard_normal(c_in).astype(np.float32), (0.5 + g.random(c_in)).astype(np.float32)
    net = qtt.NN(ctx, c_in, width, depth, p)
    net.set_scaling(shift, scale, 0.5)
    xs = torch.tensor((x.astype(np.float64) - shift[None, :, None, None]) * scale[None, :, None, None])
    pt = torch.tensor(p, dtype=torch.float64)
    assert rel(net.predict(x), 0.5 * N.forward(pt, xs, c_in, width, depth).numpy()) < 1e-5
    loss_ref, grad_ref = N.loss_and_grad(pt, xs, torch.tensor(y.astype(np.float64) / 0.5), c_in, width, depth)
    loss = net.train_step(x, y, 1e-3)
    assert abs(loss - loss_ref) <= 1e-5 * loss_ref
    assert rel(net.grad(), grad_ref.numpy()) < 1e-4
    # a second step on the same handle (buffers reused)
    assert np.isfinite(net.train_step(x, y, 1e-3))
