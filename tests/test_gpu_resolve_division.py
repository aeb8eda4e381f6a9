"""The resolve where every quotient of a back-projection is taken by division: a
coefficient of the backward map's depth row so small that, with z_min 0, a depth
could be denormal.  Against the oracle, colour exact."""
import numpy as np
import pytest

import synthetic as S
from fvv_helpers import assert_parity, gpu_run, lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("kw", [dict(), dict(pixel_weights=1), dict(hole_fill=0)])
def test_every_back_projection_by_division(oracle_mod, axis, kw):
    F = lib()
    rng = np.random.default_rng(8 + axis)
    H, W = 70, 120
    cams = S.scenes.rig_parallel(3, W, H, 90.0, 0.1)
    rgb = rng.integers(0, 256, (3, H, W, 3)).astype(np.uint8)
    dep = (1400 + 500 * np.sin(np.arange(W) / 9.0)[None, None, :] + rng.integers(0, 60, (3, H, W))).astype(np.uint16)
    dep[rng.random((3, H, W)) < 0.15] = 0
    view = cams[1].copy()
    view.t = view.t + np.array([0.03, 0.01, 0.05])
    view.R = view.R.copy()
    view.R[axis, 2] = 1e-23
    kw = dict(z_min=0.0, **kw)
    opts = F.fvv_default_options(**kw)
    _, N, _ = F.fvv_view_params(F.rig(cams, np.zeros(3)), opts, view)
    c = np.abs(np.asarray(N).reshape(3, -1)[:, 8 + axis])
    assert ((c > 0) & (c < 2.0 ** -70)).any()            # the rounding's tolerance is infinite
    g = gpu_run(cams, rgb, dep, [view], np.zeros(3), opts=opts)[0]
    ref = oracle_mod.synthesize(cams, rgb, dep, view, np.zeros(3), **kw)
    info = assert_parity(g, ref, "tiny coefficient")
    assert info["exact_rgb_fraction"] == 1.0
