"""unigs_plan.sort_passes is the number of radix passes that the binning runs."""
import pytest

from paper_2510_12174_gb300 import abi
from paper_2510_12174_gb300 import rasterizer as rz
from paper_2510_12174_gb300 import scenes


# 0, 2, 9, 10, 18 and 19 bits of a tile id
@pytest.mark.parametrize("size, n_cams, passes", [
    ((16, 16), 1, 4), ((32, 32), 1, 5), ((512, 256), 1, 5), ((513 * 16, 16), 1, 6),
    ((16384, 4096), 1, 6), ((16384, 4097), 1, 7)])
def test_sort_passes(size, n_cams, passes):
    g = abi.unigs_gaussians()
    g.n, g.sh_degree, g.n_sem, g.feat_dtype = 10, 0, 0, 0
    cams = rz.make_cameras([scenes.front_camera(*size, 100.0)] * n_cams)
    plan = abi.unigs_plan()
    assert abi.unigs_plan_init(plan, g, cams, n_cams, None, 0) == abi.UNIGS_OK
    assert plan.sort_passes == passes
    # init, culling, splats, digits, passes, emission (two for images of more
    # than 64 tiles), ranges, schedule, 3 forward, 3 backward
    big = plan.n_tiles // n_cams > 64
    assert abi.unigs_launches_per_step(plan) == 3 + 1 + passes + 1 + big + 2 + 3 + 3
