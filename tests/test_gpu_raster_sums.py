"""How the raster backward adds up a Gaussian's 2D gradients: each pixel's own
terms, and one sum per tile.

A Gaussian's position and covariance gradients are sums over pixels of
dp (v0, v1, v0^2 / 2, v0 v1, v1^2 / 2). Where v1 nearly vanishes (along the
conjugate direction of a long thin Gaussian) the last two are small differences
of large numbers unless v1 is formed per pixel, and a tile's sum must meet the
other tiles' as one number, or cancelling parts of it cost their low bits."""
import numpy as np
import pytest
import torch

from paper_2509_25191_gb300 import _lib, synth
from paper_2509_25191_gb300.autograd import Rasterizer

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -24


def _backward(rast, views, proj, image, up, use_last=True):
    g2d = torch.empty(views.num_slots(), _lib.GS_GRAD2D_FLOATS, device="cuda")
    _lib.gs_rasterize_bwd(views, rast.cfg, proj, rast.bins, image, up, g2d, rast.status, use_last=use_last)
    torch.cuda.synchronize()
    rast.check_status()
    return g2d.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("use_last", [True, False])
@pytest.mark.parametrize("tile", [(8, 8), (16, 8), (16, 16), (32, 8), (32, 16), (32, 32)])
def test_one_pixel_gives_a_rank_one_covariance_gradient(tile, use_last):
    """With one pixel's upstream gradient the (a, b, c) gradients are
    dp (v0^2 / 2, v0 v1, v1^2 / 2), so 4 a c = b^2: a and c carry two
    roundings each and b two (twice in its square), eight half-ulps in all,
    however small v1 is against v0."""
    sc = synth.uniform_box_scene(7, 600, log_scale_mu=-2.2, log_scale_sigma=0.9, sh_degree=0)
    vw = synth._views(np.concatenate([np.eye(3).reshape(-1), np.zeros(3)]), 90.0, 96, 80, 0, sc.n)
    g, views = _lib.Gaussians.from_scene(sc), _lib.Views.from_synth(vw)
    rast = Rasterizer(tile=tile)
    image, proj = rast.forward(g, views)
    seen = thin = 0
    for px, py in [(48, 40), (3, 77), (31, 31), (64, 16), (90, 8), (20, 55)]:
        up = torch.zeros(3, 80, 96, device="cuda")
        up[:, py, px] = torch.tensor([1.0, -0.5, 0.25], device="cuda")
        g2d = _backward(rast, views, proj, image, up.reshape(-1), use_last)
        a, b, c = g2d[:, 2], g2d[:, 3], g2d[:, 4]
        # (products below 1e-30 may have lost bits to the float32 range)
        on = (np.abs(a) > 1e-30) & (np.abs(c) > 1e-30) & (np.abs(b) > 1e-30)
        seen += int(on.sum())
        thin += int((np.abs(c[on] / a[on]) < 1e-3).sum())
        off = np.abs(4 * a[on] * c[on] / b[on] ** 2 - 1)
        assert off.max() <= 10 * EPS, ((px, py), off.max() / EPS)
    assert seen > 50 and thin > 5
