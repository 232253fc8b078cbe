"""Infinities in the network: what pads a convolution's operands is zero on both sides, so
that an infinite activation reaches the outputs whose stencil holds it and no others."""
import numpy as np
import pytest

import oracle.unet as U
import paper_1303_0625_gb300 as G
from test_gpu_unet import _flat

pytestmark = pytest.mark.gpu


def _ones(names, taps):
    """A network of two levels of which each named layer passes its listed input channels
    on to channel 0, through the centre tap or the sum of all nine."""
    p = {k: np.zeros_like(v) for k, v in U.init_params(2, 8).items()}
    for name, channels in names.items():
        for c in channels:
            w = p[name + ".w"]
            w[0, c, 1, 1] = 1.0
            if taps == 9:
                w[0, c] = 1.0
    p["head.w"][:, 0] = 1.0
    return p


@pytest.mark.parametrize("H,W", [(12, 20), (8, 140)])
@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_infinity_in_the_input_stays_in_its_stencil(H, W, value):
    p = _ones({"enc0a": [0], "enc0b": [0], "dec0a": [16], "dec0b": [0]}, 1)
    net = G.UNet(H, W, levels=2, base=8, max_batch=2)
    net.set_params(_flat(p, 2, 8).astype(np.float32))
    x = np.zeros((2, 8, H, W), np.float32)
    x[:, 0] = np.random.default_rng(3).integers(1, 256, (2, H, W)) / 256.0  # exact in BF16
    at = (5, 9)
    x[0, 0][at] = value
    y = net.forward(x)
    far = np.ones((2, H, W), bool)
    far[0, at[0] - 1:at[0] + 2, at[1] - 1:at[1] + 2] = False
    for o in range(3):
        assert np.array_equal(y[:, o][far], x[:, 0][far])
        if value == np.inf:
            assert y[0, o][at] == np.inf


@pytest.mark.parametrize("H,W", [(12, 20), (8, 140)])
def test_infinity_passes_an_odd_number_of_channel_groups(H, W):
    """The decoder's first convolution reads three groups of 8 channels and one of zeros."""
    p = _ones({"enc0a": [0], "enc0b": [0], "enc1a": [0], "enc1b": [0], "dec0a": [0, 16], "dec0b": [0]}, 9)
    net = G.UNet(H, W, levels=2, base=8, max_batch=1)
    net.set_params(_flat(p, 2, 8).astype(np.float32))
    x = np.full((1, 8, H, W), 0.5, np.float32)
    x[0, 0, 5, 9] = np.inf
    y = net.forward(x)
    assert (y[0, :, 5, 9] == np.inf).all()
