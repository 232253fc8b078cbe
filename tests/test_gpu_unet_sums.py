"""Sums of the network that come out the same on every run: a training step adds its
gradients in a fixed order, whichever block ends first, so that training repeats bit for
bit."""
import numpy as np
import pytest

from test_gpu_unet import _case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("levels,base,H,W,B", [
    (2, 8, 4, 6, 1),       # one split, less than a tile
    (2, 8, 10, 130, 2),    # planes as one row; 3 channel groups
    (3, 16, 12, 192, 2),   # rows in two runs
    (4, 32, 64, 128, 8),   # more splits than fit the SMs at once
])
def test_training_repeats_bit_for_bit(levels, base, H, W, B):
    net, p, x, t, fl = _case(levels, base, H, W, B, 5 * levels + W)
    start = net.params()
    loss, g = net.gradients(x, t, fl)
    for _ in range(4):
        again, h = net.gradients(x, t, fl)
        assert again == loss and np.array_equal(g, h)
    runs = []
    for _ in range(3):
        net.set_params(start)
        runs.append(([net.train_step(x, t, fl, 1e-3) for _ in range(3)], net.params()))
    for losses, params in runs[1:]:
        assert losses == runs[0][0] and np.array_equal(params, runs[0][1])
