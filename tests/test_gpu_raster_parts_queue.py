"""Images in parts of tiles where the parts outnumber the resident blocks: the
blocks take them from the queue, in the order of the sort first and of the
recorded replay lengths from the second forward on. The image is the 16x16
tiles' bit for bit, and the record that the next order comes from holds each
tile's longest replay."""
import numpy as np
import pytest
import torch

from paper_2509_25191_gb300 import _lib, synth
from paper_2509_25191_gb300.autograd import Rasterizer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile,batch", [((32, 32), (2, 1)), ((32, 32), (1, 2)), ((32, 16), (2, 1)), ((32, 16), (4, 1))])
@pytest.mark.parametrize("size", [(1000, 821), (700, 640)])
def test_parts_from_the_queue_equal_whole_tiles(size, tile, batch):
    W, H = size
    sc = synth.uniform_box_scene(6, 30_000, sh_degree=1)
    vw = synth._views(np.concatenate([np.eye(3).reshape(-1), np.zeros(3)]), float(W), W, H, 0, sc.n)
    g, views = _lib.Gaussians.from_scene(sc), _lib.Views.from_synth(vw)
    want, _ = Rasterizer(tile=(16, 16)).forward(g, views)
    rast = Rasterizer(tile=tile, batch=batch)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for _ in range(3):
        image, _ = rast.forward(g, views)
        parts = rast.bins.n_tiles * (tile[0] * tile[1] // 256)
        assert 4 * sms < parts and rast.bins.n_tiles < 16 * sms   # a queue, and a recorded order
        assert torch.equal(image, want)
        # a tile's record: the largest end of its pixels, from the start of its list
        ranges = rast.bins.tile_ranges.cpu().numpy()[:2 * rast.bins.n_tiles].reshape(-1, 2)
        last = rast.bins.last_contrib.cpu().numpy().reshape(H, W)
        work = rast.bins.tile_work.cpu().numpy()[:rast.bins.n_tiles]
        gx = -(-W // tile[0])
        for t in range(0, rast.bins.n_tiles, 7):
            x, y = t % gx * tile[0], t // gx * tile[1]
            assert work[t] == last[y:y + tile[1], x:x + tile[0]].max() - ranges[t, 0]
