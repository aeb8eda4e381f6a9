"""Layered synthesis at the edges of the BG crack pass's 64 x 4 tiles and of its
border form (views one to three pixels a side), against the oracle.  Keys,
holes, depth and colour exact."""
import pytest

import synthetic as S
from fvv_helpers import assert_parity, gpu_run, lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lay():
    return S.workload("layered_9cam_1280x720", scale=0.26)


@pytest.mark.parametrize("W,H", [(1, 1), (2, 2), (3, 3), (1, 9), (63, 4), (64, 5), (65, 3), (129, 8)])
def test_sizes(oracle_mod, lay, W, H):
    view = lay["views"][60].copy()
    s = W / view.width
    view.fx, view.fy, view.cx, view.cy = view.fx * s, view.fy * s, W / 2.0, H / 2.0
    view.width, view.height = W, H
    g = gpu_run(lay["cams"], lay["rgb"], lay["depth"], [view], lay["look_at"],
                opts=lib().fvv_default_options(layered=1), bg=lay["bg"])[0]
    ref = oracle_mod.synthesize_layered(lay["cams"], lay["rgb"], lay["depth"], lay["bg"], view, lay["look_at"])
    info = assert_parity(g, ref, "%dx%d" % (W, H))
    assert info["exact_rgb_fraction"] == 1.0
