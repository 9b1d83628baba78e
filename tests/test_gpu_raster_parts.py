"""Tiles of more than 256 pixels are rasterized in 16x16 parts whose blocks
pack the Gaussians that reach them: more of them than a batch holds, none at
all, and parts that lie outside a ragged image. The image is the 16x16 tiles'
bit for bit and the 2D gradients differ only in the order of their additions;
the L1 loss is summed over all blocks."""
import numpy as np
import pytest
import torch

from paper_2509_25191_gb300 import _lib, synth
from paper_2509_25191_gb300.autograd import Rasterizer
from tests.gpu_util import image_errors, oracle_forward, split

pytestmark = pytest.mark.gpu


def _scene(n_dense):
    # a sparse scene, and n_dense small Gaussians in front of one 16x16 part of the image
    sc = synth.uniform_box_scene(4, 300, sh_degree=1)
    dense = synth.uniform_box_scene(5, n_dense, lo=(-0.28, -0.28, 2.0), hi=(-0.14, -0.14, 3.0), log_scale_mu=-4.5,
                                    logit_sigma=0.5, sh_degree=1)
    dense.opacity_logits[:] -= 3.0   # faint: the part's pixels do not saturate early
    both, _ = synth.concat_scenes([sc, dense])
    return both


def _run(sc, vw, tile, batch, target):
    g, views = _lib.Gaussians.from_scene(sc), _lib.Views.from_synth(vw)
    rast = Rasterizer(tile=tile, batch=batch)
    image, proj = rast.forward(g, views)
    g2d = torch.empty(views.num_slots(), _lib.GS_GRAD2D_FLOATS, device="cuda")
    loss = torch.empty(1, device="cuda")
    _lib.gs_rasterize_bwd_l1(views, rast.cfg, proj, rast.bins, image, target, loss, g2d)
    torch.cuda.synchronize()
    rast.check_status()
    return image, g2d.cpu().numpy().astype(np.float64), float(loss.item())


@pytest.mark.parametrize("n_dense", [0, 127, 129, 2000])
@pytest.mark.parametrize("size", [(33, 17), (128, 96), (70, 45)])
def test_parts_equal_whole_tiles(n_dense, size):
    W, H = size
    sc = _scene(n_dense) if n_dense else synth.uniform_box_scene(4, 5, sh_degree=1)
    vw = synth._views(np.concatenate([np.eye(3).reshape(-1), np.zeros(3)]), 100.0, W, H, 0, sc.n)
    target = torch.rand(3 * W * H, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    ref_img, ref_g, _ = _run(sc, vw, (16, 16), (2, 1), target)
    worst, _ = image_errors(split(ref_img, vw), oracle_forward(sc, vw))
    assert worst <= 1e-4
    want = float((ref_img.double() - target.double()).abs().mean())
    for tile, batch in [((32, 32), (1, 1)), ((32, 32), (2, 2)), ((32, 32), (4, 1)), ((32, 16), (2, 1)),
                        ((32, 16), (1, 2))]:
        img, g2d, loss = _run(sc, vw, tile, batch, target)
        assert torch.equal(img, ref_img), (tile, batch)
        # float32 sums of the same terms in another order (each block's part, then the blocks')
        assert np.linalg.norm(g2d - ref_g) <= 1e-5 * np.linalg.norm(ref_g), (tile, batch)
        assert abs(loss - want) <= 1e-6 * want, (tile, batch)
