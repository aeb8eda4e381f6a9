"""The resolve kernel at the edges of its work split -- 64-pixel blocks, the two
pixels of a lane, bands of rows, camera groups of one to four --
on the tallest view, and where every back-projection is rounded by division,
against the oracle.  Keys, holes and depth exact, colour exact."""
import numpy as np
import pytest

import synthetic as S
from fvv_helpers import assert_parity, gpu_run, lib

pytestmark = pytest.mark.gpu


def _frames(rng, n, H, W):
    rgb = rng.integers(0, 256, (n, H, W, 3)).astype(np.uint8)
    z = 1400 + 500 * np.sin(np.arange(W) / 9.0)[None, None, :] + rng.integers(0, 60, (n, H, W))
    z[rng.random((n, H, W)) < 0.15] = 0
    return rgb, z.astype(np.uint16)


@pytest.mark.parametrize("n,W,H", [(1, 1, 1), (2, 31, 3), (3, 32, 1), (4, 33, 2), (5, 63, 4), (6, 64, 5), (7, 65, 7),
                                   (9, 127, 2), (3, 129, 6), (2, 640, 9)])
@pytest.mark.parametrize("kw", [dict(), dict(hole_fill=0), dict(pixel_weights=1)])
def test_block_band_and_group_edges(oracle_mod, n, W, H, kw):
    rng = np.random.default_rng(W * H + n)
    cams = S.scenes.rig_arc(n, 40.0, 1.5, 80, 48, 70.0)
    rgb, dep = _frames(rng, n, 48, 80)
    view = S.scenes.arc_view(7.0, 1.45, W, H, max(20.0, 70.0 * W / 80))
    g = gpu_run(cams, rgb, dep, [view], np.zeros(3), opts=lib().fvv_default_options(**kw))[0]
    ref = oracle_mod.synthesize(cams, rgb, dep, view, np.zeros(3), **kw)
    info = assert_parity(g, ref, "%d cameras, %dx%d" % (n, W, H))
    assert info["exact_rgb_fraction"] == 1.0


def test_tallest_view(oracle_mod):
    rng = np.random.default_rng(5)
    cams = S.scenes.rig_arc(2, 10.0, 1.5, 40, 30, 40.0)
    rgb, dep = _frames(rng, 2, 30, 40)
    view = S.scenes.arc_view(1.0, 1.5, 2, 65535, 40.0)
    view.fy = 40.0 * 65535 / 30
    g = gpu_run(cams, rgb, dep, [view], np.zeros(3))[0]
    ref = oracle_mod.synthesize(cams, rgb, dep, view, np.zeros(3))
    assert (ref["keys_raw"] != np.uint64(0xFFFFFFFFFFFFFFFF)).sum() > 50
    assert_parity(g, ref, "2x65535")


def test_every_quotient_by_division(oracle_mod):
    """A map whose depth row holds a coefficient near 1e-25, with z_min 0, leaves
    the range of the division-free rounding (a depth could be denormal)."""
    rng = np.random.default_rng(6)
    cams = S.scenes.rig_parallel(3, 120, 70, 90.0, 0.1)
    rgb, dep = _frames(rng, 3, 70, 120)
    view = cams[1].copy()
    view.t = view.t + np.array([0.03, 0.01, 0.05])
    view.R = view.R.copy()
    view.R[2, 0] = 1e-23
    kw = dict(z_min=0.0)
    g = gpu_run(cams, rgb, dep, [view], np.zeros(3), opts=lib().fvv_default_options(**kw))[0]
    ref = oracle_mod.synthesize(cams, rgb, dep, view, np.zeros(3), **kw)
    info = assert_parity(g, ref, "tiny coefficient")
    assert info["exact_rgb_fraction"] == 1.0


@pytest.mark.parametrize("n", [3, 4, 6, 7])
def test_many_rows_in_flight(oracle_mod, n):
    """Batches whose bands outnumber two per SM: the form of two cameras at a time."""
    rng = np.random.default_rng(40 + n)
    cams = S.scenes.rig_arc(n, 40.0, 1.5, 80, 48, 70.0)
    rgb, dep = _frames(rng, n, 48, 80)
    views = [S.scenes.arc_view(-9.0 + 2.0 * i, 1.45, 97, 131, 80.0) for i in range(10)]
    for kw in (dict(), dict(pixel_weights=1)):
        gs = gpu_run(cams, rgb, dep, views, np.zeros(3), opts=lib().fvv_default_options(**kw))
        for i in (0, 9):
            ref = oracle_mod.synthesize(cams, rgb, dep, views[i], np.zeros(3), **kw)
            info = assert_parity(gs[i], ref, "%d cameras, view %d" % (n, i))
            assert info["exact_rgb_fraction"] == 1.0
