"""Tick uploads and the depth filter on rows padded so that every wide access is
aligned while the row's end is ragged: the wide forms' own ragged ends, and for the
filter the wide staging between neighbouring tiles.  The padding holds other
values, none of which may be taken in or, on the output, overwritten."""
import numpy as np
import pytest

import synthetic as S
from oracle import jbf as J
from fvv_helpers import lib

pytestmark = pytest.mark.gpu


def _up(n, k):
    return -(-n // k) * k


def _rows(a, pitch):
    """The rows of `a` (..., H, bytes) `pitch` bytes apart on the device, 171 between them."""
    import torch
    b = np.full(a.shape[:-1] + (pitch,), 171, np.uint8)
    b[..., :a.shape[-1]] = a
    return torch.from_numpy(b).cuda()


@pytest.mark.parametrize("W", [5, 66, 259])
def test_tick_upload(W):
    """A tick uploaded from the device, seen from each camera's own pose, is that camera's frame."""
    import torch
    F = lib()
    H, n = 6, 3
    rng = np.random.default_rng(W)
    cams = S.scenes.rig_arc(n, 60.0, 1.5, W, H, 0.8 * W + 4)
    rgb = rng.integers(0, 256, (n, H, W, 3)).astype(np.uint8)
    dep = rng.integers(900, 3000, (n, H, W)).astype(np.uint16)
    rp, dp = _up(3 * W, 4), _up(2 * W, 8)
    r, d = _rows(rgb.reshape(n, H, 3 * W), rp), _rows(dep.view(np.uint8).reshape(n, H, 2 * W), dp)
    ctx = F.fvv_create(F.rig(cams, np.zeros(3)), F.fvv_default_options(crack_filter=0, hole_fill=0))
    try:
        F.fvv_upload_frames(ctx, r, H * rp, rp, d, H * dp, dp, 0)
        for k in range(n):
            out = torch.zeros((H, W, 3), dtype=torch.uint8, device="cuda")
            z = torch.zeros((H, W), dtype=torch.float32, device="cuda")
            F.fvv_synthesize(ctx, cams[k], out, W * 3, F.aux(depth=z))
            torch.cuda.synchronize()
            assert np.array_equal(out.cpu().numpy(), rgb[k]), k
            assert np.array_equal(z.cpu().numpy(), dep[k].astype(np.float32)), k
    finally:
        F.fvv_destroy(ctx)


@pytest.mark.parametrize("W,radius", [(w, r) for w in (63, 130, 261) for r in (1, 2, 3)] +
                         [(w, r) for w in (65, 131) for r in (4, 7)])
def test_filter(W, radius):
    import torch
    F = lib()
    H = 35
    rng = np.random.default_rng(W * H + radius)
    d = rng.integers(1000, 4000, (H, W)).astype(np.uint16)
    d[rng.random((H, W)) < 0.3] = 0
    d[rng.random((H, W)) < 0.05] = 65535
    rgb = (rng.integers(0, 40, (H, W, 3)) + 100 * (np.arange(W) > W // 2)[None, :, None]).astype(np.uint8)
    rp, dp = _up(3 * W, 16), _up(2 * W, 16)
    r, src = _rows(rgb.reshape(H, 3 * W), rp), _rows(d.view(np.uint8).reshape(H, 2 * W), dp)
    out = torch.full((H, dp), 205, dtype=torch.uint8, device="cuda")
    F.fvv_depth_jbf(r, rp, src, dp, out, dp, W, H, F.fvv_default_options(jbf_radius=radius, jbf_min_valid=2))
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    assert np.array_equal(got[:, :2 * W].copy().view(np.uint16), J.jbf(d, rgb, radius=radius, min_valid=2))
    assert (got[:, 2 * W:] == 205).all()
