"""The network where its kernels change over: layers just above 2^19 outputs, whose tiles of 8 x 32 pixels
and 32 channels are cut by odd grids and channel counts, just below (one thread per output), and weight
gradients on both sides of 4096 pixels and of 2^21 multiply-adds, against the float64 oracle.  Relative
error of sums of up to 18 000 products <= sqrt(18 000) eps32 ~ 8e-6; 1e-5 (outputs) and 1e-4 (gradients,
whose terms cancel) as in the tests of the whole network."""
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
    (5, 33, 3, 4, 65, 67), (3, 40, 3, 2, 91, 75), (2, 31, 3, 4, 65, 65), (4, 8, 3, 1, 64, 64), (4, 8, 3, 1, 64, 65),
    (2, 15, 3, 1, 32, 32), (2, 16, 3, 1, 32, 33)])
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
