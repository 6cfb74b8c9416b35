"""Binning at the edges of its dispatch: the radix passes' chunk sizes, the
number of tile passes, rectangles above the mask size, against the oracle's
lists (bit-exact)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2510_12174_gb300 import rasterizer as rz
from paper_2510_12174_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as ge
    ge.build()
    torch.cuda.set_device(0)


# (scene, capacity): a capacity of 4M instances and more takes the large chunks
CASES = {
    "one_gaussian": (dict(n=1, width=64, height=48, seed=1), 0),
    "one_tile": (dict(n=300, width=16, height=16, seed=2), 0),
    "two_tiles": (dict(n=2048, width=32, height=16, seed=3), 0),
    "chunk_plus_one": (dict(n=2049, width=100, height=76, seed=4), 0),
    "one_9_bit_pass": (dict(n=4000, width=512, height=256, seed=5), 0),
    "two_5_bit_passes": (dict(n=4000, width=513, height=256, seed=6), 0),
    "large_rectangles": (dict(n=1500, width=640, height=400, seed=7, log_scale_mean=-0.7), 0),
    "large_chunks": (dict(n=20000, width=333, height=251, seed=8, n_cams=3), 4_000_001),
}


@pytest.mark.parametrize("case", list(CASES))
def test_lists_match_the_oracle(case):
    kw, capacity = CASES[case]
    sc, cams = scenes.small_room(n_sem=4, **kw)
    r = rz.Renderer(rz.DeviceScene.from_scene(sc), cams, capacity=capacity)
    for _ in range(2):  # the second binning finds the first one's state
        r.preprocess_and_sort()
        keys, vals, ranges = r.sorted_instances()
        ref = oracle.bin_cameras_fast(sc, cams)
        assert np.array_equal(keys, ref["keys"])
        assert np.array_equal(vals, ref["vals"])
        assert np.array_equal(ranges, ref["ranges"])


def test_large_depth_chunks():
    """4.2M (camera, Gaussian) pairs: the depth passes take the large chunks.
    The lists are sorted by (tile, depth, index), and every pair appears once
    per kept tile."""
    sc, _ = scenes.small_room(n=70_000, width=64, height=48, n_sem=0, seed=9)
    cams = scenes.orbit_cameras(60, seed=9, resolutions=[(64, 48)])
    r = rz.Renderer(rz.DeviceScene.from_scene(sc), cams)
    r.preprocess_and_sort()
    keys, vals, ranges = r.sorted_instances()
    order = np.lexsort((vals, keys))
    assert np.array_equal(order, np.arange(len(keys)))
    off = r.plan.off[4]
    total = 60 * r.scene.n
    touched = r.ws[off: off + 4 * total].view(torch.int32).cpu().numpy()
    tiles = (keys >> np.uint64(32)).astype(np.int64)
    cam = np.searchsorted([r.plan.tile_offset[k] for k in range(60)], tiles, side="right") - 1
    assert np.array_equal(np.bincount(cam * r.scene.n + vals, minlength=total), touched)
    assert np.array_equal(np.bincount(tiles, minlength=len(ranges)),
                          ranges[:, 1].astype(np.int64) - ranges[:, 0])
