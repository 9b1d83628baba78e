"""One process may use the shared-memory batches of a tile in any order: a
smaller batch does not take the kernels' shared memory from a larger one."""
import pytest
import torch

from paper_2509_25191_gb300 import _lib, synth
from paper_2509_25191_gb300.autograd import Rasterizer

pytestmark = pytest.mark.gpu


def test_a_smaller_batch_after_a_larger_one():
    sc, vw = synth.orbit_views(0, 3000, 1, 96, 64, 100.0)
    g, views = _lib.Gaussians.from_scene(sc), _lib.Views.from_synth(vw)
    images = []
    for batch in ((4, 2), (1, 1), (2, 1), (4, 2)):
        rast = Rasterizer(tile=(32, 32), batch=batch)
        image, proj = rast.forward(g, views)
        rast.backward(g, views, proj, image, torch.ones_like(image))
        torch.cuda.synchronize()
        rast.check_status()
        images.append(image)
    assert all(torch.equal(i, images[0]) for i in images)
