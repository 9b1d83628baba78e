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


@pytest.mark.parametrize("use_last", [True, False])
@pytest.mark.parametrize("tile", [(16, 16), (32, 16), (32, 32)])
def test_a_tile_adds_one_sum(tile, use_last):
    """A round Gaussian on the centre of the middle tile column, one large
    upstream gradient of each sign at mirrored pixels of its tiles: equal
    weights, so these tiles' colour sums cancel to exactly 0 before they leave
    the tile. What is left are the single pixels of the other tiles, whose sum in
    any order is within (n - 1) half-ulps of their absolute sum; added in
    parts, the large terms would cost them seventeen bits."""
    tw, th = tile
    W, H = 3 * tw, 96
    sc = synth.uniform_box_scene(0, 1, sh_degree=0)
    sc.means[:] = (0.0, 0.0, 2.0)
    sc.log_scales[:] = np.log(1.0)
    sc.quats[:] = (1.0, 0.0, 0.0, 0.0)
    sc.opacity_logits[:] = 0.0
    vw = synth._views(np.concatenate([np.eye(3).reshape(-1), np.zeros(3)]), 60.0, W, H, 0, 1)
    g, views = _lib.Gaussians.from_scene(sc), _lib.Views.from_synth(vw)
    rast = Rasterizer(tile=tile)
    image, proj = rast.forward(g, views)
    rng = np.random.default_rng(5)
    pairs = np.zeros((3, H, W), np.float32)
    single = []
    for ty in range(H // th):
        # mirrored columns of the middle tile column, both of one row
        y, d = ty * th + int(rng.integers(th)), int(rng.integers(tw // 4, tw // 2))
        pairs[:, y, W // 2 + d] = 131072.0
        pairs[:, y, W // 2 - 1 - d] = -131072.0
        for tx in (0, 2):
            up = np.zeros((3, H, W), np.float32)
            up[:, ty * th + int(rng.integers(th)), tx * tw + int(rng.integers(tw))] = rng.uniform(0.5, 1.0, 3)
            single.append(up)
    dev = lambda u: torch.as_tensor(u.reshape(-1), device="cuda")
    terms = np.stack([_backward(rast, views, proj, image, dev(u), use_last)[0, 6:9] for u in single])
    assert (np.abs(terms) > 0).all()
    want, room = terms.sum(0), (len(terms) - 1) * EPS * np.abs(terms).sum(0)
    for _ in range(8):
        got = _backward(rast, views, proj, image, dev(pairs + np.sum(single, 0)), use_last)[0, 6:9]
        assert (np.abs(got - want) <= room).all(), (got, want, room)
