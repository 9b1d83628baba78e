"""rasterize(): an instance count above the planned capacity is found while the
raster kernel runs and the image is rendered again; two backwards give separate
gradient arrays."""
import torch

import pytest

from paper_2509_25191_gb300 import _lib, synth
from paper_2509_25191_gb300.autograd import Rasterizer, rasterize

pytestmark = pytest.mark.gpu


def test_growing_lists_and_separate_gradients():
    sc, vw = synth.orbit_views(1, 4000, 2, 120, 80, 120.0)
    g = _lib.Gaussians.from_scene(sc)
    vm = torch.as_tensor(vw.viewmats).cuda()
    intr = torch.as_tensor(vw.intrinsics).cuda()
    leaves = [t.clone().requires_grad_(True) for t in (g.means, g.log_scales, g.quats, g.opacity_logits, g.sh, vm)]
    want = rasterize(*leaves, intr, vw.width, vw.height).detach()
    rast = Rasterizer()
    rast._ensure_bins(_lib.Views.from_synth(vw), 16, "cuda")   # far too small
    image = rasterize(*leaves, intr, vw.width, vw.height, rasterizer=rast)
    assert rast.bins.capacity >= rast.last_instances > 16
    assert torch.equal(image, want)
    rast.check_status()
    up = torch.randn(image.shape, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    first = torch.autograd.grad(image, leaves, up, retain_graph=True)
    kept = [t.clone() for t in first]
    second = torch.autograd.grad(image, leaves, 2.0 * up)
    for a, k, b in zip(first, kept, second):
        assert torch.equal(a, k) and a.data_ptr() != b.data_ptr()
        # linear in the upstream gradient, up to the order of float atomics
        assert float((b - 2.0 * a).norm()) <= 1e-4 * float(b.norm())
