"""What a Rasterizer keeps after an autograd forward and backward: its tile
lists and scratch, and no parameter gradients (autograd owns those)."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2509_25191_gb300 import _lib, synth
from paper_2509_25191_gb300.autograd import Rasterizer, rasterize

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pose_only", [False, True])
def test_backward_keeps_only_lists_and_scratch(pose_only):
    sc = synth.uniform_box_scene(2, 60_000, sh_degree=3)
    f = lambda a: torch.as_tensor(np.asarray(a, np.float32)).cuda()
    leaves = [f(a).requires_grad_(not pose_only) for a in (sc.means, sc.log_scales, sc.quats, sc.opacity_logits, sc.sh)]
    vm = f([[1, 0, 0, 0, 1, 0, 0, 0, 1, 0, 0, 0]]).requires_grad_(True)
    intr = f([[80.0, 80.0, 48.0, 40.0]])

    def step(rast):
        rasterize(*leaves, vm, intr, [96], [80], rasterizer=rast).square().sum().backward()
        for t in leaves + [vm]:
            assert (t.grad is not None) == t.requires_grad
            t.grad = None

    step(Rasterizer())   # (the library and the caches are warm)
    torch.cuda.synchronize()
    before = torch.cuda.memory_allocated()
    rast = Rasterizer()
    step(rast)
    step(rast)
    torch.cuda.synchronize()
    kept = torch.cuda.memory_allocated() - before
    bins = [t for t in vars(rast.bins).values() if torch.is_tensor(t)] + [rast.status]
    blocks = int(_lib.load().gs_pose_blocks(ctypes.c_int64(sc.n)))
    want = sum(t.numel() * t.element_size() for t in bins) + 4 * (_lib.GS_GRAD2D_FLOATS * sc.n + 12 * blocks)
    # (every tensor is rounded up to 512 bytes; the five parameter gradients would be 14 MB)
    assert kept <= want + 512 * (len(bins) + 16), (kept, want)


def test_direct_and_autograd_backward_share_the_scratch():
    """Rasterizer.backward and the autograd backward in turn give what each gives
    alone (their 2D gradients are rewritten by every call)."""
    sc = synth.uniform_box_scene(2, 3000, sh_degree=1)
    f = lambda a: torch.as_tensor(np.asarray(a, np.float32)).cuda()
    leaves = [f(a).requires_grad_(True) for a in (sc.means, sc.log_scales, sc.quats, sc.opacity_logits, sc.sh)]
    vm, intr = f([[1, 0, 0, 0, 1, 0, 0, 0, 1, 0, 0, 0]]), f([[80.0, 80.0, 48.0, 40.0]])
    g = _lib.Gaussians(*(t.detach() for t in leaves))
    views = _lib.Views(vm, intr, [96], [80], [0], [sc.n])
    rast = Rasterizer()
    image, proj = rast.forward(g, views)
    up = torch.ones_like(image)
    direct, _, _ = rast.backward(g, views, proj, image, up)
    want = direct.means.clone()
    out = rasterize(*leaves, vm, intr, [96], [80], rasterizer=rast)
    means = torch.autograd.grad(out.sum(), leaves)[0]
    assert torch.equal(direct.means, want)   # the earlier call's gradients are its own
    scale = float(want.abs().max())
    # (float32 sums in another order)
    assert float((means - want).abs().max()) <= 1e-5 * scale
    assert means.data_ptr() != direct.means.data_ptr()
