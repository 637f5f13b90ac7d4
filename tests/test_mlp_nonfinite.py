"""Losses and gradients that leave the FP32 range: the loss is an FP64 sum of the
FP32 differences squared, a bias gradient the FP64 sum of its column rounded to
FP32, so what is finite in FP64 stays finite and an infinity stays one."""
import numpy as np
import pytest
import torch

from paper_1406_4254_gb300 import etics, surrogate

pytestmark = pytest.mark.gpu


def _setup(dims, batch, seed=3):
    net = surrogate.Mlp(dims, seed=seed)
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn((batch, dims[0]), generator=g, device="cuda").to(torch.bfloat16)
    t = torch.randn((batch, dims[-1]), generator=g, device="cuda")
    return net, x, t


def _parts(net, dims):
    """Weight and bias gradients per layer."""
    out, o = [], 0
    for a, b in zip(dims, dims[1:]):
        out.append((net.grads[o:o + a * b].view(a, b), net.grads[o + a * b:o + a * b + b]))
        o += a * b + b
    return out


# narrow output layer (three widths of layer behind it), general output layers
# (column sums of the layer below by a kernel of their own, in the product)
SHAPES = [([8, 64, 64, 3], 130), ([8, 256, 256, 3], 2000), ([16, 3], 131), ([8, 64, 64, 9], 130),
          ([8, 64, 64, 16], 130)]


@pytest.mark.parametrize("dims,batch", SHAPES)
@pytest.mark.parametrize("size", [1e18, 1e25, 3e38])
def test_loss_beyond_the_fp32_range_is_finite(dims, batch, size):
    net, x, t = _setup(dims, batch)
    y = net.forward(x).double()
    t[batch // 2, 1] = size
    t[1, 0] = -size
    want = ((y - t.double()) ** 2).mean().item()
    loss = net.loss_grad(x, t).item()
    # each difference is rounded to FP32 (relative 2^-24, twice that in its
    # square); the sums are FP64
    assert np.isfinite(want) and abs(loss - want) <= 2.0 ** -22 * want


@pytest.mark.parametrize("dims,batch", SHAPES)
@pytest.mark.parametrize("bad", [float("inf"), -float("inf"), float("nan")])
def test_a_nonfinite_target_reaches_loss_and_bias_gradients_as_it_is(dims, batch, bad):
    net, x, t = _setup(dims, batch)
    row, col = batch // 2, 1
    t[row, col] = bad
    loss = net.loss_grad(x, t).item()
    assert np.isnan(loss) if np.isnan(bad) else loss == float("inf")
    (w, db) = _parts(net, dims)[-1]
    others = torch.arange(dims[-1], device="cuda") != col
    assert torch.isfinite(db[others]).all()
    assert torch.isnan(db[col]) if np.isnan(bad) else db[col].item() == -bad
    if len(dims) > 2:
        # dz of that row is (y - t) w (1 - h^2): an infinity of the weight's sign
        o = net.n - dims[-1] - dims[-2] * dims[-1]
        wl = net.params_bf16[o:o + dims[-2] * dims[-1]].view(dims[-2], dims[-1])[:, col].float()
        assert (wl != 0).all()
        got = _parts(net, dims)[-2][1]
        if np.isnan(bad):
            assert torch.isnan(got).all()
        else:
            assert torch.equal(got, -bad * torch.sign(wl))
