"""D-SSIM of an image against itself, where SSIM is 1 whatever the image: the
variances and the covariance have to agree to rounding although each is a small
difference of large blurs in bright, flat regions."""
import numpy as np
import pytest
import torch

from paper_2509_25191_gb300 import _lib

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -24


@pytest.mark.parametrize("noise", [0.0, 1e-3, 0.05])
@pytest.mark.parametrize("level", [0.3, 0.77, 0.95])
@pytest.mark.parametrize("size", [(90, 70), (640, 480), (1237, 822)])   # a block per channel, few tiles, many
def test_an_image_against_itself_has_no_dssim(size, level, noise):
    """With (x - y)^2 exactly 0 the two factors of SSIM are ratios of numbers
    that differ in the last places: a value of SSIM is off by at most ten
    half-ulps (two products, two reciprocals, a sum each in l1, l2, d1, d2), and
    their mean by as much again for the sums within a tile and one half-ulp per
    tile that adds to the loss."""
    W, H = size
    gen = torch.Generator("cuda").manual_seed(W)
    x = (level + noise * torch.randn(3 * W * H, generator=gen, device="cuda")).clamp(0.0, 1.0)
    views = _lib.Views(None, None, [W], [H], [0], [0])
    loss, grad = torch.empty(3, device="cuda"), torch.empty_like(x)
    _lib.gs_l1_dssim_loss(views, x, x.clone(), loss, grad, 0.2)
    total, l1, dssim = loss.tolist()
    tiles = -(-W // 32) * -(-H // 32)
    room = (20 + min(tiles, 64)) * EPS   # (the sum's rounding grows like the root of the additions)
    assert l1 == 0.0
    assert abs(dssim) <= room, dssim / EPS
    assert abs(total - np.float32(0.2) * dssim) <= EPS
