"""Frame uploads and syntheses beside the persistent serving kernel: the kernel is
resident on every SM, and their kernels have to run beside it instead of waiting
until it returns, which it does only after idle_us without work."""
import time

import numpy as np
import pytest

import synthetic as S
from oracle import codec as K
from fvv_helpers import lib

pytestmark = pytest.mark.gpu

CODEC = dict(z_near=0.4, z_far=6.0, alpha=0.004, beta=0.995)
IDLE_MS = 400.0


# the depth filter's kernels (512 threads and 47 KB of shared memory up to radius
# 3, 36 KB at radius 7), and the decoder of rows that are no multiples of 16
@pytest.mark.parametrize("W,radius,yuv", [(320, 0, 0), (320, 3, 0), (320, 7, 0), (314, 0, 1), (314, 3, 1)])
@pytest.mark.parametrize("max_width", [640, 1920])
def test_uploads_run_beside_the_persistent_kernel(W, radius, yuv, max_width):
    """While the kernel waits for work (up to IDLE_MS) a tick is uploaded and a
    view of it is requested.  A kernel of the upload that does not fit beside it
    starts when it returns, so that would take IDLE_MS; half of that is the line,
    some fifty times what the upload and the view take.  The views equal those
    rendered alone from the same tick."""
    import torch
    F = lib()
    H, n = 180, 3
    rng = np.random.default_rng(W + radius)
    cams = S.scenes.rig_arc(n, 40.0, 1.5, W, H, 250.0)
    rgb = rng.integers(0, 256, (n, H, W, 3)).astype(np.uint8)
    dep = rng.integers(1300, 1700, (n, H, W)).astype(np.uint16)
    dep[rng.random((n, H, W)) < 0.1] = 0
    planes = [K.encode(d, unit_m=0.001, **CODEC) for d in dep]
    view = S.scenes.arc_view(7.0, 1.5, 640, 360, 500.0)
    ctx = F.fvv_create(F.rig(cams, np.zeros(3)), F.fvv_default_options(frame_slots=2, jbf_radius=radius))

    def upload(tick, turn):
        for k in range(n):
            c = np.ascontiguousarray(np.roll(rgb[k], turn, axis=0))
            if yuv:
                F.fvv_upload_frame_yuv(ctx, k, c, W * 3, *(planes[k][0], W, planes[k][1], planes[k][2], W // 2), tick)
            else:
                F.fvv_upload_frame(ctx, k, c, W * 3, dep[k], W * 2, tick)

    def image():
        return torch.zeros((360, 640 * 3), dtype=torch.uint8, device="cuda")

    try:
        if yuv:
            for k in range(n):
                F.fvv_set_depth_codec(ctx, k, F.fvv_depth_codec_default(**CODEC))
        alone, outs = [image() for _ in range(4)], [image() for _ in range(5)]
        for i in range(4):                         # (loads every kernel before the serving starts)
            upload(i, i)
            F.fvv_synthesize(ctx, view, alone[i], 640 * 3)
        torch.cuda.synchronize()
        F.fvv_serve_start(ctx, F.fvv_serve_default_cfg(lanes=2, max_batch=4, memory_budget=256 << 20, persistent=1,
                                                       max_width=max_width, idle_us=int(IDLE_MS * 1000)))
        F.fvv_serve_poll(ctx, F.fvv_serve_submit(ctx, 0, view, outs[4], 640 * 3), 5_000_000)   # the kernel runs
        ms = []
        for i in range(4):
            t0 = time.perf_counter()
            upload(4 + i, i)
            F.fvv_serve_poll(ctx, F.fvv_serve_submit(ctx, i, view, outs[i], 640 * 3), 5_000_000)
            ms.append(1e3 * (time.perf_counter() - t0))
        st = F.fvv_serve_stats(ctx)
        F.fvv_serve_stop(ctx)
        assert st["completed"] == 5 and st["failed"] == 0
        assert all(torch.equal(outs[i], alone[i]) for i in range(4)) and torch.equal(outs[4], alone[3])
        assert not torch.equal(alone[0], alone[1])
        assert max(ms) < IDLE_MS / 2, ms
    finally:
        F.fvv_destroy(ctx)


# narrow views take the resolve's wide form; the outputs that a refinement needs its largest one
@pytest.mark.parametrize("W,max_width", [(160, 160), (320, 320), (640, 640), (1280, 1280), (320, 1920)])
@pytest.mark.parametrize("aux", [0, 1])
def test_syntheses_run_beside_the_persistent_kernel(W, max_width, aux):
    """As above with a view that is synthesised directly, on a stream of its own
    (aux: with the top-3 weights and per-pixel angular weights)."""
    import torch
    F = lib()
    h, w, n = 180, 320, 3
    rng = np.random.default_rng(W)
    cams = S.scenes.rig_arc(n, 40.0, 1.5, w, h, 250.0)
    rgb = rng.integers(0, 256, (n, h, w, 3)).astype(np.uint8)
    dep = rng.integers(1300, 1700, (n, h, w)).astype(np.uint16)
    H = W // 2
    view, small = S.scenes.arc_view(7.0, 1.5, W, H, 0.78 * W), S.scenes.arc_view(3.0, 1.5, 160, 96, 125.0)
    out, alone = (torch.zeros((H, W * 3), dtype=torch.uint8, device="cuda") for _ in range(2))
    served, ref = (torch.zeros((96, 160 * 3), dtype=torch.uint8, device="cuda") for _ in range(2))
    t3 = torch.zeros((H, W, 3), dtype=torch.float32, device="cuda")
    s = torch.cuda.Stream()
    ctx = F.fvv_create(F.rig(cams, np.zeros(3)), F.fvv_default_options(pixel_weights=aux))

    def synthesise(o):
        F.fvv_synthesize(ctx, view, o, W * 3, F.aux(top3=t3) if aux else None, s)
        s.synchronize()

    try:
        for k in range(n):
            F.fvv_upload_frame(ctx, k, rgb[k], w * 3, dep[k], w * 2, 0)
        synthesise(alone)
        F.fvv_synthesize(ctx, small, ref, 160 * 3, None, s)
        s.synchronize()
        F.fvv_serve_start(ctx, F.fvv_serve_default_cfg(lanes=2, max_batch=4, memory_budget=256 << 20, persistent=1,
                                                       max_width=max_width, idle_us=int(IDLE_MS * 1000)))
        F.fvv_serve_poll(ctx, F.fvv_serve_submit(ctx, 0, small, served, 160 * 3), 5_000_000)       # the kernel runs
        t0 = time.perf_counter()
        synthesise(out)
        ms = 1e3 * (time.perf_counter() - t0)
        F.fvv_serve_stop(ctx)
        assert torch.equal(out, alone) and torch.equal(served, ref)
        assert ms < IDLE_MS / 2
    finally:
        F.fvv_destroy(ctx)
