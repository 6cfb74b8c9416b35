"""Renderer.forward with its read-back of the status block."""
import copy

import pytest
import torch

from paper_2510_12174_gb300 import abi
from paper_2510_12174_gb300 import rasterizer as rz
from paper_2510_12174_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as ge
    ge.build()
    torch.cuda.set_device(0)


def _room(seed):
    return scenes.small_room(n=3000, width=64, height=52, n_sem=12, seed=seed)


@pytest.mark.parametrize("build_inside", [False, True])
def test_first_frame_in_inference_mode(build_inside):
    """A renderer whose first frame is drawn in inference mode (an evaluation
    before training) draws the next one outside it, and the other way round."""
    sc, cams = _room(101)
    with torch.inference_mode(build_inside):
        r = rz.Renderer(rz.DeviceScene.from_scene(sc), cams)
    with torch.inference_mode():
        first = {k: v.clone() for k, v in r.forward().items()}
    for mode in (False, True):
        with torch.inference_mode(mode):
            out = r.forward()
            assert all(torch.equal(first[k], out[k]) for k in first)


def test_deep_copy_of_a_used_renderer():
    """A deep copy draws the same frame, and re-plans on its own."""
    sc, cams = _room(102)
    r = rz.Renderer(rz.DeviceScene.from_scene(sc), cams)
    out = r.forward()
    q = copy.deepcopy(r)
    capacity = r.capacity
    q._plan(64)  # overflows: the copy reads its own status block and grows
    for a in (q, r):
        again = a.forward()
        assert all(torch.equal(out[k], again[k]) for k in out)
    assert r.capacity == capacity and q.capacity > 64


def test_non_finite_parameter_leaves_the_callers_frame():
    """With the check on, a non-finite opacity raises before the caller's
    buffers are written."""
    sc, cams = _room(103)
    cfg = abi.unigs_config_default()
    cfg.flags |= abi.UNIGS_FLAG_CHECK_FINITE
    scene = rz.DeviceScene.from_scene(sc)
    r = rz.Renderer(scene, cams, cfg=cfg)
    out = r.forward()
    before = {k: v.clone() for k, v in out.items()}
    good = scene.opacity.clone()
    scene.opacity[::2] = float("nan")
    with pytest.raises(RuntimeError):
        r.forward(out)
    torch.cuda.synchronize()
    assert all(torch.equal(before[k], out[k]) for k in out)
    scene.opacity.copy_(good)
    assert all(torch.equal(before[k], v) for k, v in r.forward(out).items())


def test_overflow_on_a_side_stream():
    """A frame over the capacity is drawn again on the stream it was asked for
    on, whatever stream the first workspace came from."""
    sc, cams = _room(104)
    ref = rz.Renderer(rz.DeviceScene.from_scene(sc), cams).forward()
    r = rz.Renderer(rz.DeviceScene.from_scene(sc), cams, capacity=64)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        out = r.forward()
        assert r.capacity > 64
    side.synchronize()
    assert all(torch.equal(ref[k], out[k]) for k in ref)
