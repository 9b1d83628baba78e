"""The work order that gs_bin_sort leaves for the raster kernels: every tile
once, by decreasing count bucket, and within a bucket no run of neighbouring
tiles (they would be rasterized at the same time, and the 2D gradients of the
Gaussians that cover them would be added in another order on every run)."""
import numpy as np
import pytest
import torch

from paper_2509_25191_gb300 import _lib, synth
from paper_2509_25191_gb300.autograd import Rasterizer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [0, 40, 20_000])
@pytest.mark.parametrize("size,views", [((1600, 1066), 1), ((979, 546), 4), ((1024, 528), 1)])
def test_work_order_keeps_neighbours_apart(size, views, n):
    """Thread i of 1,024 places tiles i per, i per + 1, ..., per >= 2 here: places
    next to each other in a bucket hold tiles of different threads, or (where the
    bucket has none of the others) of one thread's later rounds. At most one place in
    ten is allowed to follow its neighbour; in ascending order nearly all do."""
    sc = synth.uniform_box_scene(1, max(n, 1), sh_degree=0)
    if not n:
        sc.means[:] = (0.0, 0.0, -1.0)   # nothing visible: one bucket
    vw = synth._views(np.tile(np.concatenate([np.eye(3).reshape(-1), np.zeros(3)]), (views, 1)), float(size[0]),
                      size[0], size[1], 0, sc.n)
    g, v = _lib.Gaussians.from_scene(sc), _lib.Views.from_synth(vw)
    rast = Rasterizer(tile=(16, 16))
    bins = rast.bin_sort(v, rast.project(g, v))
    torch.cuda.synchronize()
    T = bins.n_tiles
    assert T > 2048
    order = bins.tile_order.cpu().numpy()[:T]
    ranges = bins.tile_ranges.cpu().numpy()[:2 * T].reshape(T, 2)
    assert np.array_equal(np.sort(order), np.arange(T))
    count = (ranges[:, 1] - ranges[:, 0])[order]
    bucket = np.where(count > 0, np.floor(np.log2(np.maximum(count, 1))) + 1, 0)
    assert (np.diff(bucket) <= 0).all()
    same = np.diff(bucket) == 0
    assert (np.abs(np.diff(order))[same] == 1).mean() < 0.1
