"""Tick uploads, the depth encoder and the depth filter at the edges of their
wide-access forms: widths and pitches that leave a ragged end or no alignment,
each against the plain statement of the result."""
import numpy as np
import pytest

import synthetic as S
from oracle import codec as K
from oracle import jbf as J
from fvv_helpers import lib

pytestmark = pytest.mark.gpu

CODEC = dict(z_near=0.4, z_far=6.0, alpha=0.004, beta=0.995)


def _dev(a, pad):
    """`a`'s bytes on the device, `pad` bytes past an aligned start."""
    import torch
    b = torch.zeros(a.nbytes + pad + 64, dtype=torch.uint8, device="cuda")
    b[pad:pad + a.nbytes] = torch.from_numpy(np.frombuffer(a.tobytes(), np.uint8).copy()).cuda()
    return b, b.data_ptr() + pad


@pytest.mark.parametrize("W,H,pad", [(4, 2, 0), (6, 4, 0), (8, 6, 2), (64, 4, 0), (66, 8, 4), (130, 10, 0), (260, 6, 0)])
@pytest.mark.parametrize("yuv", [0, 1])
def test_tick_upload(W, H, pad, yuv):
    """A tick uploaded from the device, seen from each camera's own pose, is that camera's frame."""
    import torch
    F = lib()
    rng = np.random.default_rng(W + H + pad + yuv)
    n = 3
    cams = S.scenes.rig_arc(n, 60.0, 1.5, W, H, 0.8 * W + 4)
    rgb = rng.integers(0, 256, (n, H, W, 3)).astype(np.uint8)
    dep = rng.integers(900, 3000, (n, H, W)).astype(np.uint16)
    ctx = F.fvv_create(F.rig(cams, np.zeros(3)), F.fvv_default_options(crack_filter=0, hole_fill=0))
    try:
        r, rp = _dev(rgb, pad)
        if yuv:
            for k in range(n):
                F.fvv_set_depth_codec(ctx, k, F.fvv_depth_codec_default(**CODEC))
            planes = [K.encode(d, unit_m=0.001, **CODEC) for d in dep]
            frames = np.stack([np.concatenate([p.reshape(-1) for p in q]) for q in planes])
            d, dp = _dev(frames, pad)
            F.fvv_upload_frames_yuv(ctx, rp, rgb[0].nbytes, W * 3, dp, frames[0].nbytes, 0)
            want = [K.decode(*q, CODEC["z_near"], CODEC["z_far"], 0.001) for q in planes]
        else:
            d, dp = _dev(dep, pad)
            F.fvv_upload_frames(ctx, rp, rgb[0].nbytes, W * 3, dp, dep[0].nbytes, W * 2, 0)
            want = dep
        for k in range(n):
            out = torch.zeros((H, W, 3), dtype=torch.uint8, device="cuda")
            z = torch.zeros((H, W), dtype=torch.float32, device="cuda")
            F.fvv_synthesize(ctx, cams[k], out, W * 3, F.aux(depth=z))
            torch.cuda.synchronize()
            assert np.array_equal(out.cpu().numpy(), rgb[k]), k
            assert np.array_equal(z.cpu().numpy(), np.asarray(want[k], np.float32)), k
    finally:
        F.fvv_destroy(ctx)


@pytest.mark.parametrize("W,H,dpad,ypad", [(2, 2, 0, 0), (4, 2, 0, 0), (6, 4, 0, 0), (8, 2, 4, 0), (64, 6, 0, 1), (68, 4, 8, 0),
                                           (258, 4, 0, 0), (1028, 2, 0, 0)])
def test_encode(W, H, dpad, ypad):
    import torch
    F = lib()
    rng = np.random.default_rng(W + H + dpad)
    cams = S.scenes.rig_arc(1, 0.0, 1.5, W, H, 50.0)
    ctx = F.fvv_create(F.rig(cams, np.zeros(3)))
    try:
        F.fvv_set_depth_codec(ctx, 0, F.fvv_depth_codec_default(**CODEC))
        d = rng.integers(0, 7000, (H, W)).astype(np.uint16)
        d[rng.random((H, W)) < 0.2] = 0
        d[rng.random((H, W)) < 0.1] = 65535
        b, p = _dev(d, dpad)
        y = torch.zeros(H * W + 64, dtype=torch.uint8, device="cuda")
        u = torch.zeros((H // 2, W // 2), dtype=torch.uint8, device="cuda")
        v = torch.zeros_like(u)
        F.fvv_depth_encode_yuv(ctx, 0, p, W * 2, y.data_ptr() + ypad, W, u, v, W // 2)
        torch.cuda.synchronize()
        ry, ru, rv = K.encode(d, unit_m=0.001, **CODEC)
        assert np.array_equal(y[ypad:ypad + H * W].cpu().numpy().reshape(H, W), ry)
        assert np.array_equal(u.cpu().numpy(), ru) and np.array_equal(v.cpu().numpy(), rv)
    finally:
        F.fvv_destroy(ctx)


@pytest.mark.parametrize("W,H,pad", [(63, 17, 0), (64, 16, 0), (72, 33, 0), (72, 33, 2), (127, 15, 0), (200, 40, 0)])
@pytest.mark.parametrize("radius", [1, 4, 7])
def test_filter(W, H, pad, radius):
    import torch
    F = lib()
    rng = np.random.default_rng(W * H + radius)
    d = rng.integers(1000, 4000, (H, W)).astype(np.uint16)
    d[rng.random((H, W)) < 0.3] = 0
    d[rng.random((H, W)) < 0.05] = 65535
    d[5:12, 3:30] = 0                                   # a gap wider than the window
    rgb = (rng.integers(0, 40, (H, W, 3)) + 100 * (np.arange(W) > W // 2)[None, :, None]).astype(np.uint8)
    r, rp = _dev(rgb, 0)
    b, dp = _dev(d, pad)
    out = torch.full((H, W), -1, dtype=torch.int16, device="cuda")
    F.fvv_depth_jbf(rp, W * 3, dp, W * 2, out, W * 2, W, H, F.fvv_default_options(jbf_radius=radius, jbf_min_valid=2))
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy().view(np.uint16), J.jbf(d, rgb, radius=radius, min_valid=2))
