"""Binning of a frame whose large rectangles overfill the array of kept-tile
bits although its instances fit: those that found the array full are tested
again in the emission.  Against the oracle's lists (bit-exact)."""
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


def thin_diagonals(n, seed):
    """Thin splats across the whole image: rectangles of up to a thousand
    tiles, of which a diagonal band is kept."""
    rng = np.random.default_rng(seed)
    ang = np.radians(45.0 + rng.uniform(-12, 12, n)) * rng.choice([-1, 1], n)
    z = rng.uniform(2.8, 3.2, n)
    f = lambda x: np.ascontiguousarray(x, dtype=np.float32)
    return scenes.Scene(
        mean=f([rng.uniform(-0.2, 0.2, n), rng.uniform(-0.2, 0.2, n), z]),
        quat=f([np.cos(ang / 2), np.zeros(n), np.zeros(n), np.sin(ang / 2)]),
        scale=f([np.full(n, 2.0), np.full(n, 0.04), np.full(n, 0.04)]),
        opacity=f(rng.uniform(0.3, 0.9, n)), kfac=f(np.ones(n)), sh=f(rng.uniform(-1, 1, (n, 1, 3))),
        sem=f(rng.uniform(-1, 1, (n, 4))), sh_degree=0)


def test_rectangles_beyond_the_bit_array():
    sc = thin_diagonals(400, 11)
    cams = [scenes.front_camera(640, 400, 400.0)]
    ref = oracle.bin_cameras_fast(sc, cams)
    need = len(ref["keys"])
    r = rz.Renderer(rz.DeviceScene.from_scene(sc), cams, capacity=need)
    for _ in range(2):
        r.preprocess_and_sort()
        assert r.last_instances == need and r.capacity == need  # fits: no new plan
        # words asked for (byte 56 of the status block) and the array's
        o = r.plan.off[0] + 56
        assert int(r.ws[o: o + 8].view(torch.int64).item()) > need // 8 + 1024
        keys, vals, ranges = r.sorted_instances()
        assert np.array_equal(keys, ref["keys"])
        assert np.array_equal(vals, ref["vals"])
        # (an empty tile's range is empty; the oracle places it)
        some = ref["ranges"][:, 1] > ref["ranges"][:, 0]
        assert np.array_equal(ranges[some], ref["ranges"][some])
        assert np.array_equal(ranges[~some, 0], ranges[~some, 1])
