"""The network's kernels for large layers (more than 2^19 outputs and four channels; weight gradients
over more than 4096 pixels): odd sizes at the edges of their tiles against the float64 oracle, and
weights that meet no pixel of the grid, which have no effect even where they are not finite.

Tolerances as for the whole network: sums of 9 * 33 products per output and of at most 2^16 products
per weight: 1e-5 (outputs) and 1e-4 (gradients, whose terms cancel)."""
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


def params(c_in, width, depth, seed):
    g = inputs.rng(seed)
    p = []
    for co, ci in N.layer_shapes(c_in, width, depth):
        p += [g.standard_normal(co * ci * 9) * np.sqrt(2.0 / (ci * 9)), 0.1 * g.standard_normal(co)]
    return np.concatenate(p).astype(np.float32)


def rel(a, b):
    a = np.asarray(a, dtype=np.float64).ravel(); b = np.asarray(b, dtype=np.float64).ravel()
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("c_in,width,depth,B,H,W", [(3, 9, 3, 2, 211, 161), (5, 33, 3, 3, 97, 63), (4, 8, 2, 1, 1, 70001),
                                                    (2, 12, 2, 1, 45001, 1), (6, 40, 2, 1, 113, 127)])
def test_large_layers_at_odd_sizes(ctx, c_in, width, depth, B, H, W):
    from paper_2507_05222_gb300 import qtt
    g = inputs.rng(7 * width + H)
    p = params(c_in, width, depth, width + H)
    x = g.standard_normal((B, c_in, H, W)).astype(np.float32)
    y = g.standard_normal((B, 1, H, W)).astype(np.float32)
    net = qtt.NN(ctx, c_in, width, depth, p)
    pt, xt = torch.tensor(p, dtype=torch.float64), torch.tensor(x, dtype=torch.float64)
    assert rel(net.predict(x), N.forward(pt, xt, c_in, width, depth).numpy()) < 1e-5
    loss_ref, grad_ref = N.loss_and_grad(pt, xt, torch.tensor(y, dtype=torch.float64), c_in, width, depth)
    assert abs(net.train_step(x, y, 1e-3) - loss_ref) <= 1e-5 * loss_ref
    assert rel(net.grad(), grad_ref.numpy()) < 1e-4


def test_weights_outside_the_grid_are_not_applied(ctx):
    """One row of pixels: the upper and lower weights meet no pixel, whatever their values."""
    from paper_2507_05222_gb300 import qtt
    c_in, width, B, H, W = 4, 16, 1, 1, 40000
    x = inputs.rng(5).standard_normal((B, c_in, H, W)).astype(np.float32)
    y = inputs.rng(7).standard_normal((B, 1, H, W)).astype(np.float32)
    p = params(c_in, width, 3, 6)
    ref = qtt.NN(ctx, c_in, width, 3, p).predict(x)
    for bad in (np.inf, -np.inf, np.nan):
        q = p.copy()
        for o, (co, ci) in zip((0, width * (c_in * 9 + 1)), ((width, c_in), (width, width))):
            w = q[o:o + co * ci * 9].reshape(co, ci, 3, 3)
            w[:, :, 0] = bad
            w[:, :, 2] = bad
        net = qtt.NN(ctx, c_in, width, 3, q)
        assert np.array_equal(net.predict(x), ref)
        # nor in the gradient, which is that of finite weights
        good = qtt.NN(ctx, c_in, width, 3, p)
        assert net.train_step(x, y, 1e-3) == good.train_step(x, y, 1e-3)
        assert np.array_equal(net.grad(), good.grad())


def test_values_not_finite_reach_only_the_weights_they_meet(ctx):
    """A NaN in the grid's last row meets no upper weight (its output row would lie outside): those weights have
    the gradient of the finite neighbours, the units that the NaN reaches being off (ReLU).  H and W are not
    multiples of the tiles'."""
    from paper_2507_05222_gb300 import qtt
    c_in, width, B, H, W = 3, 12, 2, 97, 61
    g = inputs.rng(11)
    p = params(c_in, width, 2, 12)
    x = g.standard_normal((B, c_in, H, W)).astype(np.float32)
    y = g.standard_normal((B, 1, H, W)).astype(np.float32)
    x[0, 1, H - 1, 20] = np.nan
    x[1, 1, H - 1, 0] = np.nan
    net = qtt.NN(ctx, c_in, width, 2, p)
    net.train_step(x, y, 1e-3)
    n0 = width * c_in * 9
    dw = net.grad()[:n0].reshape(width, c_in, 3, 3)
    pt = torch.tensor(p, dtype=torch.float64, requires_grad=True)
    w0, b0 = pt[:n0].view(width, c_in, 3, 3), pt[n0:n0 + width]
    w1, b1 = pt[n0 + width:-1].view(1, width, 3, 3), pt[-1:]

    def conv(t, w, b):
        t = torch.nn.functional.pad(t, (1, 1, 0, 0), mode="circular")
        return torch.nn.functional.conv2d(torch.nn.functional.pad(t, (0, 0, 1, 1)), w, b)

    xt = torch.tensor(x, dtype=torch.float64)
    fine = torch.where(torch.isfinite(xt), xt, torch.zeros_like(xt))
    hit = conv((~torch.isfinite(xt)).double().sum(1, keepdim=True), torch.ones(1, 1, 3, 3, dtype=torch.float64), None)
    out = conv(torch.relu(conv(fine, w0, b0)) * (hit == 0), w1, b1)
    loss = ((out - torch.tensor(y, dtype=torch.float64)) ** 2).mean()
    (grad,) = torch.autograd.grad(loss, pt)
    ref = grad[:n0].view(width, c_in, 3, 3).numpy()
    assert np.isfinite(dw[:, 1, 0]).all()
    assert not np.isfinite(dw[:, 1, 1:]).any()
    assert rel(dw[:, 1, 0], ref[:, 1, 0]) < 1e-4
