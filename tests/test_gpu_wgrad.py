"""Weight gradients across the edges of the 128-pixel tiles and of the rows that
the blocks share out."""
import numpy as np
import pytest
import torch

from paper_2301_13601_gb300 import surrogate as S
from test_gpu_surrogate import SCALE, make_inputs, random_params

pytestmark = pytest.mark.gpu


def gradient(p, q, n, qt):
    nimg, _, H, W = q.shape
    with S.Surrogate(H, W, nimg=nimg, out_scale=SCALE, train=True) as sur:
        sur.set_params(p)
        return sur.loss_grad(*(torch.as_tensor(np.ascontiguousarray(a), device="cuda") for a in (q, n, qt)),
                             want_loss=True, want_grad=True)[1].astype(np.float64)


# a row per block and less, two and three tiles, images that blocks share, several ring turns per block
@pytest.mark.parametrize("nimg, H, W", [(1, 3, 256), (3, 5, 384), (1, 1, 1280), (2, 300, 256)])
def test_gradient_does_not_depend_on_where_the_tiles_lie(nimg, H, W):
    """The network is periodic and every pixel is computed alike, so rolling all
    inputs leaves the terms of every weight's sum as they are; only their order
    changes. At most 1e6 FP32 additions in chains of 1e4 steps of relative 2^-23,
    on sums whose terms cancel to about 1e-2 of their size: below 1e-3. A column
    of a tile taken from the wrong pixel is off by about sqrt(1/128) = 9e-2."""
    p = random_params(11)
    q, n = make_inputs(nimg, H, W, 12)
    qt = q + 0.05 * np.random.default_rng(13).standard_normal(q.shape).astype(np.float32)
    ref = gradient(p, q, n, qt)
    for dy, dx in ((0, 1), (1, 0), (H // 2, 64), (0, -1)):
        got = gradient(p, *(np.roll(a, (dy, dx), axis=(2, 3)) for a in (q, n, qt)))
        for ws, _, bs in S.param_slices():
            for sl in (ws, bs):
                assert np.linalg.norm(got[sl] - ref[sl]) < 1e-3 * np.linalg.norm(ref[sl]), (dy, dx, sl)
