"""The network's convolutions where their tiling changes: images a pixel
column short of, at and past the width of a tile with its neighbours (one run
of pixels or three row segments per channel group), fewer pixels than a tile,
several tiles per block, channel counts with an odd number of groups of 8 (a
zero group), weights held or streamed, and a batch below max_batch on planes
that a larger one has used.

The oracle rounds what it stores going forward to BF16, as the GPU does: on a
few pixels a ReLU that a rounding turns on or off is a large part of a gradient
(0.3 of the smallest case's with an unrounded oracle).

Tolerances: every layer between input and result rounds to BF16 (2^-9
relative at most, FP32 sums); 3 levels have 10 such layers forward and back
(2e-2), 4 levels 14 (3e-2 for gradients)."""
import numpy as np
import pytest

import oracle.unet as U
import paper_1303_0625_gb300 as G
from test_gpu_unet import _bf16, _case, _rel, _unflat

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("levels,base,H,W,B", [
    (2, 8, 4, 6, 1),      # less than a tile
    (2, 8, 6, 126, 1),    # padded rows of 128: one run of pixels
    (2, 8, 6, 128, 2),    # padded rows of 130: three segments of a full tile
    (2, 8, 10, 130, 2),   # rows and tiles out of step; 3 groups and a zero one
    (3, 16, 12, 260, 1),  # 6 and 12 groups; N of 96 backward
    (3, 16, 12, 192, 2),  # weight gradient: rows in two runs, one, two rows to a run of three
    (4, 32, 64, 128, 5),  # streamed weights; more tiles than resident blocks
])
def test_tile_edges(levels, base, H, W, B, monkeypatch):
    relu, pool = U.relu, U.pool
    monkeypatch.setattr(U, "relu", lambda v: _bf16(relu(v)))
    monkeypatch.setattr(U, "pool", lambda v: _bf16(pool(v)))
    net, p, x, t, fl = _case(levels, base, H, W, B, 3 * levels + W)
    y_ref, cache = U.forward(p, x, levels, keep=True)
    y = net.forward(x)
    assert _rel(y, y_ref) <= 2e-2
    loss_ref, dy = U.loss(y_ref, t, fl)
    g_ref = U.backward(p, cache, dy, levels)
    loss, g = net.gradients(x, t, fl)
    assert abs(loss - loss_ref) <= 2e-2 * loss_ref
    gv = _unflat(g, levels, base)
    for k in g_ref:
        assert _rel(gv[k], g_ref[k]) <= (3e-2 if levels == 4 else 2e-2), (k, _rel(gv[k], g_ref[k]))


@pytest.mark.parametrize("levels,base,H,W", [(2, 8, 10, 130), (4, 16, 24, 64)])
def test_smaller_batches_leave_nothing_behind(levels, base, H, W):
    net, p, x, t, fl = _case(levels, base, H, W, 5, 2)
    one = G.UNet(H, W, levels=levels, base=base, max_batch=2)
    one.set_params(net.params())
    first = net.forward(x)
    assert np.array_equal(net.forward(x[:2]), one.forward(x[:2]))
    assert np.array_equal(net.forward(x), first)
    la, ga = net.gradients(x[3:], t[3:], fl[3:])
    lb, gb = one.gradients(x[3:], t[3:], fl[3:])
    assert abs(la - lb) <= 1e-6 * abs(lb)  # sums of FP32 in another order
    assert _rel(ga, gb) <= 1e-5
