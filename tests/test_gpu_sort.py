"""The on-chip sort of a tile (gs_bin_sort): sizes around a block, a vector of
buckets and the on-chip limit, and depths that fill its bins and buckets
unevenly, against the unique (depth, slot) order."""
import numpy as np
import pytest
import torch

from paper_2509_25191_gb300 import _lib
from paper_2509_25191_gb300.autograd import Rasterizer

pytestmark = pytest.mark.gpu


def _depths(kind, n, rng):
    if kind == "uniform":
        return rng.uniform(0.3, 11.0, n)
    if kind == "clustered":   # most keys in a sliver of the range, one far away
        d = 5.0 + 1e-3 * rng.standard_normal(n)
        d[0] = 1e6
        return d
    if kind == "nearly equal":   # a few float32 steps: many keys per bucket, ties by slot
        return 2.0 + 2.4e-7 * rng.integers(0, 3, n)
    if kind == "two values":
        return np.where(rng.random(n) < 0.5, 0.5, 3e38)
    return np.full(n, 1.5)


@pytest.mark.parametrize("kind", ["uniform", "clustered", "nearly equal", "two values", "equal"])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 33, 511, 512, 513, 2047, 2048, 2049, 4093, 4095, 4096, 4097, 9001])
def test_one_tile_is_in_depth_slot_order(kind, n):
    rng = np.random.default_rng(n)
    depth = _depths(kind, n, rng).astype(np.float32)
    proj = np.zeros((n, _lib.GS_RECORD_FLOATS), np.float32)
    proj[:, 0:2] = 8.0    # every record reaches the one 16x16 tile
    proj[:, 2:4] = 1.0
    proj[:, 11] = 1.0
    proj[:, 14] = depth
    views = _lib.Views(torch.zeros(1, 12, device="cuda"), torch.ones(1, 4, device="cuda"), [16], [16], [0], [n])
    rast = Rasterizer()
    bins = rast.bin_sort(views, torch.as_tensor(proj).cuda())
    torch.cuda.synchronize()
    rast.check_status()
    order = np.lexsort((np.arange(n), depth))
    assert bins.tile_ranges.cpu().numpy().tolist() == [0, n]
    assert (bins.ids.cpu().numpy()[:n].astype(np.uint32) == order).all()
    want = depth[order].view(np.uint32).astype(np.uint64) << np.uint64(32) | order.astype(np.uint64)
    assert (bins.keys.cpu().numpy()[:n].view(np.uint64) == want).all()
