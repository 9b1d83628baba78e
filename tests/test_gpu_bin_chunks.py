"""Binning in smaller chunks (few slots), the work order over several rounds of
tiles, and the launches left out for small images: against the oracle's lists,
and two forwards and backwards on the same lists give the same image and
gradients."""
import numpy as np
import pytest
import torch

from paper_2509_25191_gb300 import _lib, synth
from paper_2509_25191_gb300.autograd import Rasterizer
from tests.gpu_util import gpu_forward, image_errors, oracle_forward, split

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 511, 513, 1025, 4097, 20000])
@pytest.mark.parametrize("size,tile", [((40, 24), (16, 16)), ((640, 480), (16, 16)), ((1000, 700), (8, 8)),
                                       ((300, 260), (32, 32))])
def test_lists_cover_every_instance_in_order(n, size, tile):
    W, H = size
    sc = synth.uniform_box_scene(n, n)
    eye = np.concatenate([np.eye(3).reshape(-1), np.zeros(3)])
    vw = synth._views(np.stack([eye, eye]), 0.9 * W, W, H, 0, n)
    g, views = _lib.Gaussians.from_scene(sc), _lib.Views.from_synth(vw)
    rast = Rasterizer(tile=tile)
    proj = rast.project(g, views)
    bins = rast.bin_sort(views, proj)
    torch.cuda.synchronize()
    rast.check_status()
    p = proj.cpu().numpy()
    T, slots = views.num_tiles(rast.cfg), np.nonzero(p[:, 2] > 0)[0]
    f = np.float32
    lo = lambda c, e, t, m: np.clip(np.floor((p[slots, c] - p[slots, e]) / f(t)), 0, m).astype(np.int64)
    hi = lambda c, e, t, m: np.clip(np.floor((p[slots, c] + p[slots, e]) / f(t)) + 1, 0, m).astype(np.int64)
    Gx, Gy = -(-W // tile[0]), -(-H // tile[1])
    x0, x1, y0, y1 = lo(0, 2, tile[0], Gx), hi(0, 2, tile[0], Gx), lo(1, 3, tile[1], Gy), hi(1, 3, tile[1], Gy)
    per = np.maximum(x1 - x0, 0) * np.maximum(y1 - y0, 0)
    counts = np.zeros(T, np.int64)
    for k in np.nonzero(per)[0]:
        base = (slots[k] // n) * Gx * Gy
        for y in range(y0[k], y1[k]):
            counts[base + y * Gx + x0[k]:base + y * Gx + x1[k]] += 1
    ends = np.cumsum(counts)
    ranges = bins.tile_ranges.cpu().numpy().reshape(-1, 2)[:T]
    assert (ranges[:, 1] == ends).all() and (ranges[:, 0] == ends - counts).all()
    order = bins.tile_order.cpu().numpy()[:T]
    assert (np.sort(order) == np.arange(T)).all()
    keys = bins.keys.cpu().numpy()[:ends[-1] if T else 0].view(np.uint64)
    inside = np.ones(len(keys), bool)
    inside[ranges[:, 0][counts > 0]] = False   # a tile's first key has no predecessor in it
    assert (keys[1:] > keys[:-1])[inside[1:]].all()


@pytest.mark.parametrize("size,tile", [((96, 64), (16, 16)), ((640, 480), (16, 16)), ((640, 480), (32, 32)),
                                       ((96, 64), (32, 16))])
def test_repeated_rasterization_on_the_same_lists(size, tile):
    W, H = size
    sc = synth.uniform_box_scene(3, 2500, sh_degree=1)
    vw = synth._views(np.concatenate([np.eye(3).reshape(-1), np.zeros(3)]), 0.9 * W, W, H, 0, sc.n)
    rast, g, views, image, proj = gpu_forward(sc, vw, tile=tile)
    worst, _ = image_errors(split(image, vw), oracle_forward(sc, vw))
    assert worst <= 1e-4
    up = torch.randn(views.num_image_floats(), device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    first = None
    for _ in range(3):
        img = torch.full_like(image, float("nan"))
        _lib.gs_render_fwd(views, rast.cfg, proj, rast.bins, img, rast.status)
        g2d = torch.empty(views.num_slots(), _lib.GS_GRAD2D_FLOATS, device="cuda")
        _lib.gs_rasterize_bwd(views, rast.cfg, proj, rast.bins, img, up, g2d, rast.status)
        torch.cuda.synchronize()
        rast.check_status()
        first = g2d if first is None else first
        assert torch.equal(img, image)
        assert float((g2d - first).norm()) <= 1e-5 * float(first.norm())
