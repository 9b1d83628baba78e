"""The mean L1 loss that the raster backward folds in, at every shape of launch:
a block per tile or fewer, with and without an ordering kernel before it, with
and without the forward's record, and again on the same lists."""
import numpy as np
import pytest
import torch

from paper_2509_25191_gb300 import _lib, synth
from paper_2509_25191_gb300.autograd import Rasterizer
from paper_2509_25191_gb300.step import GraphStep

pytestmark = pytest.mark.gpu


def _inputs(W, H):
    sc = synth.uniform_box_scene(3, 300, sh_degree=0)
    vw = synth._views(np.concatenate([np.eye(3).reshape(-1), np.zeros(3)]), float(W), W, H, 0, sc.n)
    g, views = _lib.Gaussians.from_scene(sc), _lib.Views.from_synth(vw)
    target = torch.rand(3 * W * H, device="cuda", generator=torch.Generator("cuda").manual_seed(W + H))
    return g, views, target


def _room(want, sms):
    # up to two blocks per SM add to the loss one after another, each addition off by
    # at most half an ulp of the sum; above that the order is a tree's
    return 2 * sms * 2.0 ** -24 * want


# rows of one tile per SM each: the image has SMs x rows tiles
@pytest.mark.parametrize("tile,rows", [((8, 8), r) for r in (1, 2, 8, 9, 15, 16, 18, 20, 21, 32, 33)] +
                         [((16, 8), r) for r in (1, 2, 8, 9, 14, 15, 16)] +
                         [((16, 16), r) for r in (1, 2, 4, 5, 8, 9)] + [((32, 8), r) for r in (2, 5, 8)] +
                         [((32, 16), r) for r in (1, 2, 3, 4, 5)] + [((32, 32), r) for r in (1, 2, 3, 5)])
def test_folded_l1_loss_at_every_launch_size(tile, rows):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    a = next(k for k in (8, 4, 2, 1) if sms % k == 0)   # a squarer image of as many tiles
    W, H = tile[0] * sms // a, tile[1] * rows * a
    g, views, target = _inputs(W, H)
    rast = Rasterizer(tile=tile)
    image, proj = rast.forward(g, views)
    assert rast.bins.n_tiles == sms * rows
    want = float((image.double() - target.double()).abs().mean())
    g2d = torch.empty(views.num_slots(), _lib.GS_GRAD2D_FLOATS, device="cuda")
    loss = torch.empty(1, device="cuda")
    for use_last in (True, True, False, False):
        loss.fill_(7.0)
        _lib.gs_rasterize_bwd_l1(views, rast.cfg, proj, rast.bins, image, target, loss, g2d, rast.status,
                                 use_last=use_last)
        assert abs(float(loss.item()) - want) <= _room(want, sms), (use_last, float(loss.item()), want)
    rast.check_status()


@pytest.mark.parametrize("tile,size", [((8, 8), (400, 400)), ((8, 8), (512, 304)), ((16, 8), (640, 240)),
                                       ((32, 32), (640, 416)), ((32, 32), (416, 416))])
def test_captured_step_reports_the_mean_absolute_difference(tile, size):
    g, views, target = _inputs(*size)
    step = GraphStep(g, views, target, tile=tile)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for _ in range(3):
        step.replay()
        torch.cuda.synchronize()
        want = float((step.image.double() - target.double()).abs().mean())
        assert abs(float(step.loss.item()) - want) <= _room(want, sms)
