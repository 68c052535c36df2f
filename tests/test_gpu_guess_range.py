"""The learned guess's loss and its gradient at the ends of the binary32 range.
All weights but the last layer's biases are zero, so that the output u is one
constant; loss = 1 - |<u, t>|^2 / (|u|^2 |t|^2) does not depend on u's size."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
SHAPES = [("W1", 16 * 256), ("b1", 256), ("W2", 256 * 8192), ("b2", 8192), ("W3", 32 * 128), ("b3", 16), ("W4", 16 * 64),
          ("b4", 8), ("W5", 64), ("b5", 2)]
AT = {}
_o = 0
for _n, _k in SHAPES:
    AT[_n] = slice(_o, _o + _k)
    _o += _k


def gradient(lib, u, targets, batch):
    net = lib.GuessNet(seed=0)
    w = torch.zeros(net.num_params, dtype=torch.float32, device="cuda")
    w[AT["b4"]] = 1.0
    w[AT["b5"].start] = u
    net.set_params(w)
    feats = torch.zeros((batch, 8), dtype=torch.float32, device="cuda")
    g, loss = net.grad(feats, targets)
    return g.cpu().numpy(), float(loss.item())


def quarter(batch):
    """t = 1 at the points of even x and y, 0 elsewhere: loss 3/4, and with N = 65536
    points dL/d Re u = -3 / (2 B u N) at those points, 1 / (2 B u N) at the others."""
    t = torch.zeros((batch, 16, 64, 64), dtype=torch.complex128, device="cuda")
    t[:, :, ::2, ::2] = 1.0
    return t


@pytest.mark.parametrize("batch", [1, 4])
@pytest.mark.parametrize("u", [1.0, 1e34, 4e-39])
def test_gradient_over_the_binary32_range(lib, batch, u):
    """u = 1e34 has gradients of 2e-39 (subnormal), u = 4e-39 is subnormal itself.
    dL/dW5 at the even points is the sum over 16384 B rows of bf16 operands (2^-8,
    and 2^-133 where they are subnormal: 0.04 here): 6%."""
    g, loss = gradient(lib, u, quarter(batch), batch)
    assert abs(loss - 0.75) <= 1e-6
    dW5 = g[AT["W5"]].reshape(8, 4, 2)  # [input channel][position (y, x)][Re, Im]
    u = float(np.float32(u))
    for pos in range(4):
        want = (-1.5 if pos == 0 else 0.5) / (65536.0 * u) * 16384.0
        assert np.all(np.abs(dW5[:, pos, 0] - want) <= 0.06 * abs(want)), (pos, dW5[:, pos, 0], want)


def test_nan_gradient_stays_nan(lib):
    """A zero target has no overlap to normalise by: 0 / 0 in loss and gradient."""
    g, loss = gradient(lib, 1.0, 0.0 * quarter(2), 2)
    assert np.isnan(loss) and np.isnan(g[AT["W5"]].reshape(8, 4, 2)[:, :, 0]).all() and np.isnan(g[AT["b5"]]).all()
