"""The rounding of the semantic gradient's sum over a tile.

A training run amplifies it: Adam's first steps have the size of the learning
rate whatever the gradient's, the logits are then rounded to bfloat16, and the
next iteration sees every logit that crossed a rounding boundary.  So the sum
keeps its order: the hi and lo parts of the weights meet in one accumulator,
16 pixels at a time.  On an image of one tile each gradient is the sum of two
partials (a channel's hi and lo rows), the same bits in either order, and is
compared with the bits of the kernel that fixed this order.
"""
import base64
import json
import os

import numpy as np
import pytest
import torch

from paper_2510_12174_gb300 import abi
from paper_2510_12174_gb300 import rasterizer as rz
from paper_2510_12174_gb300 import scenes

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(__file__), "golden", "sem_grad_one_tile.json")


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as ge
    ge.build()
    torch.cuda.set_device(0)


def sem_gradient(n, n_sem, seed):
    """dL/d(logits) of n Gaussians in front of a 16x16 image, from inputs that
    are multiples of powers of two (exact on every machine)."""
    rng = np.random.default_rng(seed)

    def draw(shape, lo, hi, unit):
        return (rng.integers(int(lo / unit), int(hi / unit), size=shape) * unit).astype(np.float32)

    z = draw(n, 2, 6, 2.0 ** -10)
    xy = draw((2, n), -0.4375, 0.4375, 2.0 ** -10) * z
    sc = scenes.Scene(mean=np.concatenate([xy, z[None]]), quat=draw((4, n), -1, 1, 2.0 ** -8),
                      scale=draw((3, n), 0.0625, 0.75, 2.0 ** -8),
                      opacity=draw(n, 0.0625, 0.75, 2.0 ** -8), kfac=draw(n, 0.5, 1, 2.0 ** -8),
                      sh=draw((n, 1, 3), -1, 1, 2.0 ** -6), sem=draw((n, n_sem), -2, 2, 2.0 ** -4),
                      sh_degree=0, feat_bf16=True)
    r = rz.Renderer(rz.DeviceScene.from_scene(sc), [scenes.front_camera(16, 16, 16.0)])
    assert abi.unigs_plan_paths(r.plan) & abi.UNIGS_PATH_BWD_TC
    out = r.forward()
    up = torch.from_numpy(draw(n_sem * 256, -1, 1, 2.0 ** -12)).cuda()
    g = r.backward(out, {"logits": up})["sem"].cpu().numpy()
    assert r.status()[0] == abi.UNIGS_OK
    return g


@pytest.mark.parametrize("n_sem", [12, 24, 40])
def test_bits_of_the_semantic_gradient(n_sem):
    with open(GOLDEN) as f:
        ref = np.frombuffer(base64.b64decode(json.load(f)[str(n_sem)]), "<f4").reshape(-1, n_sem)
    got = sem_gradient(len(ref), n_sem, seed=n_sem)
    assert np.count_nonzero(ref) > ref.size // 2
    assert np.array_equal(got.view(np.uint32), ref.view(np.uint32))
