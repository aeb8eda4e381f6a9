"""Performance cases of the view-synthesis library.

Each case is one thing that a user of the library has it do, through the
public entry points of ``paper_2007_00558_gb300.fvv``: views synthesised one
at a time or in batches, a live tick taken in and shown, many viewers served,
the depth codec, the depth pre-filter, and the refinement network's inference
and training.  Sizes are those of the library's own workloads (2 cameras
320x240, 9 cameras 1280x720 on a 90 degree arc, 18 cameras 1920x1080 on a 180
degree arc, 128x128 training crops); drawn cases spread over the same ranges,
odd and ragged sizes among them.  Frames are ray-cast on the GPU from seeded
scenes of spheres in front of a checkered cylinder wall and floor, with 1 %
depth noise and about 5 % of the depth missing in blobs, as the library's
synthetic workloads have them.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2007_00558_gb300.fvv as F

DEPTH_BG = 65535
Z_FAR = 8000.0
_stream = None


def stream():
    """The one stream all calls go to, as a render loop has it."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _views(name, cams, w, h, vw, vh, views, n_ref=0, layered=False, pixel_weights=False, aux=False, arc=90.0):
    return {"name": name, "kind": "views", "cams": cams, "w": w, "h": h, "vw": vw, "vh": vh, "views": views,
            "n_ref": n_ref, "layered": layered, "pixel_weights": pixel_weights, "aux": aux, "arc": arc}


def listed():
    return [
        # the smallest call: one small view from two cameras, where launches and host work count
        _views("view_320x240_2cam", 2, 320, 240, 320, 240, 1, arc=6.0),
        # an interactive viewer: one view of the newest tick from all nine cameras
        _views("view_1280x720_9cam", 9, 1280, 720, 1280, 720, 1),
        # the throughput workload: 32 views, each of its own tick, all cameras as references
        _views("batch32_1280x720_9cam", 9, 1280, 720, 1280, 720, 32),
        # the largest rig at full HD with the three nearest references weighted per
        # pixel, and the depth and hole outputs that a compositor takes
        _views("batch8_1920x1080_18cam_3ref", 18, 1920, 1080, 1920, 1080, 8, n_ref=3, pixel_weights=True, aux=True,
               arc=180.0),
        # layered foreground / background synthesis
        _views("layered8_1280x720_9cam", 9, 1280, 720, 1280, 720, 8, layered=True),
        # a live tick: YUV420 depth frames taken in (decoded, packed, pre-filtered) and one view shown from it
        {"name": "tick_yuv_jbf_1280x720_9cam", "kind": "tick", "cams": 9, "w": 1280, "h": 720, "vw": 1280, "vh": 720,
         "n_ref": 3, "yuv": True, "radius": 3},
        # sixteen viewers' requests of mixed resolution through the serving loop
        {"name": "serve16_mixed_9cam", "kind": "serve", "cams": 9, "w": 1280, "h": 720, "viewers": 16},
        # the transmission chain's depth codec: a tick encoded camera by camera, decoded in one call
        {"name": "codec_1280x720_9cam", "kind": "codec", "cams": 9, "w": 1280, "h": 720},
        # the depth pre-filter on one frame of a ragged size
        {"name": "jbf_1274x717", "kind": "jbf", "w": 1274, "h": 717, "radius": 3},
        # refinement of a batch of views, bf16 network at its default widths
        {"name": "refine_bf16_4x1280x720", "kind": "refine", "n": 4, "w": 1280, "h": 720, "w1": 32, "w2": 64, "w3": 128,
         "e4m3": False},
        # refinement with the quantised wide network
        {"name": "refine_e4m3_wide_2x640x360", "kind": "refine", "n": 2, "w": 640, "h": 360, "w1": 48, "w2": 96,
         "w3": 192, "e4m3": True},
        # gradients of one training batch of crops
        {"name": "train_8x128x128", "kind": "train", "n": 8, "w": 128, "h": 128, "w1": 32, "w2": 64, "w3": 128},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["view", "view", "batch", "batch", "batch", "layered", "tick", "serve", "codec", "jbf", "refine",
                       "refine", "train"])
    if kind in ("view", "batch", "layered"):
        cams = rng.randint(2, 18)
        w = _log(rng, 200, 1920)
        h = max(16, int(w * rng.uniform(0.5, 0.8)))
        vw = _log(rng, 200, 1920)
        vh = max(16, int(vw * rng.uniform(0.5, 0.8)))
        views = 1 if kind == "view" else _log(rng, 2, 32)
        c = {"kind": "views", "cams": cams, "w": w, "h": h, "vw": vw, "vh": vh, "views": views,
             "n_ref": rng.choice([0, 0, min(3, cams), rng.randint(1, cams)]), "layered": kind == "layered",
             "pixel_weights": rng.random() < 0.3, "aux": rng.random() < 0.3, "arc": 180.0 if cams > 9 else 90.0}
        # no more work than the throughput workload (pixels of every camera of every view; the
        # layered and per-pixel-weight forms do more for each)
        cap = 32 * 9 * 2 * 1280 * 720 // (2 if c["layered"] or c["pixel_weights"] else 1)
        c["views"] = max(1, min(views, cap // (2 * cams * max(w * h, vw * vh))))
        return c
    if kind == "tick":
        w = 2 * _log(rng, 100, 960)
        h = 2 * max(8, int(w * rng.uniform(0.25, 0.4)))
        return {"kind": "tick", "cams": rng.randint(2, 12), "w": w, "h": h, "vw": _log(rng, 200, 1920),
                "vh": _log(rng, 150, 1080), "n_ref": rng.choice([0, 2]), "yuv": rng.random() < 0.5,
                "radius": rng.choice([0, 2, 3])}
    if kind == "serve":
        w = _log(rng, 320, 1920)
        return {"kind": "serve", "cams": rng.randint(3, 12), "w": w, "h": int(w * 0.5625), "viewers": _log(rng, 4, 32)}
    if kind == "codec":
        w = 2 * _log(rng, 100, 960)
        return {"kind": "codec", "cams": rng.randint(1, 18), "w": w, "h": 2 * max(8, int(w * rng.uniform(0.25, 0.4)))}
    if kind == "jbf":
        w = _log(rng, 200, 1920)
        return {"kind": "jbf", "w": w, "h": max(16, int(w * rng.uniform(0.5, 0.8))), "radius": rng.randint(1, 5)}
    widths = rng.choice([(32, 64, 128), (48, 96, 192), (32, 64, 128), (64, 96, 128)])
    c = {"n": rng.randint(1, 4), "w": 4 * _log(rng, 30, 320), "w1": widths[0], "w2": widths[1], "w3": widths[2]}
    c["h"] = 4 * max(8, int(c["w"] * rng.uniform(0.125, 0.18)))
    if kind == "train":
        c.update(kind="train", n=rng.randint(1, 8), w=4 * _log(rng, 16, 80))
        c["h"] = 4 * max(8, int(c["w"] * rng.uniform(0.125, 0.25)))
    else:
        c.update(kind="refine", e4m3=rng.random() < 0.5)
    # no more work than the listed refinement of four 1280x720 views (training: forward and two backward passes)
    px = 4 * 1280 * 720 * 112896 // sum(9 * a * b // d for (a, b), d in zip(_net_layers(c), _SCALE))
    c["n"] = max(1, min(c["n"], px // ((3 if kind == "train" else 1) * c["w"] * c["h"])))
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _look(center, w, h, f):
    """Pinhole camera at `center` looking at the origin (world y points down)."""
    c = np.asarray(center, float)
    z = -c / np.linalg.norm(c)
    x = np.cross([0.0, 1.0, 0.0], z)
    x /= np.linalg.norm(x)
    R = np.stack([x, np.cross(z, x), z])
    return SimpleNamespace(width=w, height=h, fx=f, fy=f, cx=(w - 1) / 2.0, cy=(h - 1) / 2.0, R=R, t=-R @ c)


def _on_arc(deg, radius, y, w, h):
    a = math.radians(deg)
    return _look([radius * math.sin(a), y, -radius * math.cos(a)], w, h, 0.78125 * w)


def _rig(n, arc, w, h):
    radius = 1.5 if n <= 9 else 2.0
    angles = [0.0] if n == 1 else [arc * (i / (n - 1) - 0.5) for i in range(n)]
    return [_on_arc(a, radius, 0.0, w, h) for a in angles], radius


def _swing(n, arc, radius, w, h, gen):
    """Views along a swing within the arc, from a random phase."""
    p = float(torch.rand((), generator=gen))
    return [F.camera(_on_arc(0.25 * arc * math.sin(2 * math.pi * (p + i / 37.0)), radius, -0.05, w, h))
            for i in range(n)]


def _scene(gen):
    return [(torch.rand(3, generator=gen) * torch.tensor([1.6, 0.7, 1.6]) - torch.tensor([0.8, 0.45, 0.8]),
             0.05 + 0.2 * float(torch.rand((), generator=gen)), 40 + 200 * torch.rand(3, generator=gen))
            for _ in range(16)]


def _raycast(cam, scene):
    """(colour [H, W, 3] float, z [H, W] metres, foreground [H, W]) on the GPU."""
    dev = "cuda"
    R = torch.tensor(cam.R, dtype=torch.float32, device=dev)
    o = torch.tensor(-cam.R.T @ cam.t, dtype=torch.float32, device=dev)
    u = (torch.arange(cam.width, device=dev, dtype=torch.float32) - cam.cx) / cam.fx
    v = (torch.arange(cam.height, device=dev, dtype=torch.float32) - cam.cy) / cam.fy
    d = torch.stack([u[None, :].expand(cam.height, -1), v[:, None].expand(-1, cam.width),
                     torch.ones(cam.height, cam.width, device=dev)], -1) @ R
    a = d[..., 0] ** 2 + d[..., 2] ** 2
    b = o[0] * d[..., 0] + o[2] * d[..., 2]
    z = (-b + torch.sqrt(torch.clamp(b * b - a * (o[0] ** 2 + o[2] ** 2 - 16.0), min=0))) / a
    floor_z = (0.5 - o[1]) / d[..., 1]
    on_floor = (floor_z > 0) & (floor_z < z)
    z = torch.where(on_floor, floor_z, z)
    p = o + z[..., None] * d
    s = torch.where(on_floor, torch.floor(p[..., 0] / 0.25) + torch.floor(p[..., 2] / 0.25),
                    torch.floor(torch.atan2(p[..., 0], p[..., 2]) * 8) + torch.floor(p[..., 1] / 0.5))
    dark = (s.long() % 2 == 0)[..., None]
    rgb = torch.where(dark, torch.tensor([70.0, 80.0, 95.0], device=dev), torch.tensor([190.0, 180.0, 160.0], device=dev))
    fg = torch.zeros_like(on_floor)
    dd = (d * d).sum(-1)
    light = torch.tensor([-0.41, -0.41, -0.82], device=dev)
    for c, r, col in scene:
        oc = o - c.to(dev)
        bb = d @ oc
        disc = bb * bb - dd * (oc @ oc - r * r)
        t = (-bb - torch.sqrt(torch.clamp(disc, min=0))) / dd
        hit = (disc > 0) & (t > 0.05) & (t < z)
        z = torch.where(hit, t, z)
        fg = fg | hit
        n = (oc + t[..., None] * d) / r
        lam = 0.2 + 0.8 * torch.clamp(n @ light, min=0)
        rgb = torch.where(hit[..., None], lam[..., None] * col.to(dev), rgb)
    return rgb, z, fg


def _gaps(n, h, w, gen):
    """Masks [n, h, w] of missing depth: blobs over about 5 % of each frame."""
    low = torch.rand(n, 1, max(2, h // 8), max(2, w // 8), device="cuda", generator=gen)
    f = torch.nn.functional.interpolate(low, size=(h, w), mode="bilinear", align_corners=False)[:, 0]
    cut = torch.quantile(f.reshape(n, -1)[:, :: max(1, h * w // 100000)], 0.05, dim=1)
    return f < cut[:, None, None]


class _Frames:
    """Clean renders of a rig, and noisy ticks of them."""

    def __init__(self, cams, seed):
        self.gen = torch.Generator().manual_seed(int(seed))
        self.dgen = torch.Generator(device="cuda").manual_seed(int(seed))
        scene = _scene(self.gen)
        r = [_raycast(c, scene) for c in cams]
        self.rgb = torch.stack([x[0] for x in r])
        self.mm = torch.stack([x[1] for x in r]) * 1000.0
        self.fg = torch.stack([x[2] for x in r])

    def tick(self, layered=False):
        """(rgb uint8 [K, H, W, 3], depth codes int16 [K, H, W]) of one capture tick."""
        K, H, W = self.mm.shape
        rgb = (self.rgb + 4.0 * torch.randn(K, H, W, 1, device="cuda", generator=self.dgen)).clamp(0, 255)
        d = torch.round(self.mm * (1 + 0.01 * torch.randn(K, H, W, device="cuda", generator=self.dgen)))
        d = d.clamp(1, 65534).int()
        d[_gaps(K, H, W, self.dgen)] = 0
        if layered:
            d[~self.fg] = DEPTH_BG
        return rgb.round().to(torch.uint8).contiguous(), d.to(torch.int16).contiguous()


def _yuv(depth):
    """Dense planar YUV420 depth frames [K, H*W*3/2] of codes [K, H, W] (z_near 0.3 m, z_far 10 m)."""
    K, H, W = depth.shape
    z = (depth.int() & 0xFFFF).double() / 1000.0
    y = torch.floor(4093.0 * (1.0 / z.clamp(min=1e-3) - 0.1) / (1.0 / 0.3 - 0.1) + 2.5).int()
    y = torch.where((z >= 0.3) & (z <= 10.0), y, torch.ones_like(y))
    lsb, msb = y & 255, y >> 8
    luma = torch.where((msb & 1) == 1, 255 - lsb, lsb)

    def pair(m):
        a, b = m[..., 0::2], m[..., 1::2]
        return sum((((a >> i) & 1) << (2 * i)) | (((b >> i) & 1) << (2 * i + 1)) for i in range(4))

    return torch.cat([luma.reshape(K, -1), pair(msb[:, 0::2]).reshape(K, -1), pair(msb[:, 1::2]).reshape(K, -1)],
                     1).to(torch.uint8).contiguous()


class _State:
    """A context with its buffers; gives the context back when dropped."""

    def __init__(self, case, cams, **opts):
        self.case, self.look = case, [0.0, 0.0, 0.0]
        self.ctx = F.fvv_create(F.rig(cams, self.look), F.fvv_default_options(**opts))
        self.s = stream()

    def __del__(self):
        if getattr(self, "ctx", None):
            F.fvv_destroy(self.ctx)
            self.ctx = None


def _upload(st, tick, rgb, depth):
    K, H, W = depth.shape
    F.fvv_upload_frames(st.ctx, rgb, H * W * 3, W * 3, depth, H * W * 2, W * 2, tick, st.s)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("refine", "train"):
        st = _prepare_net(case, seed)
    elif kind == "jbf":
        st = SimpleNamespace(case=case, s=stream())
        rgb, depth = _Frames([_on_arc(0.0, 1.5, 0.0, case["w"], case["h"])], seed).tick()
        st.rgb, st.depth = rgb[0].contiguous(), depth[0].contiguous()
        st.out = torch.zeros_like(st.depth)
        st.opt = F.fvv_default_options(jbf_radius=case["radius"])
    else:
        st = _prepare_rig(case, seed)
    torch.cuda.synchronize()
    return st


def _prepare_rig(case, seed):
    kind, K, w, h = case["kind"], case["cams"], case["w"], case["h"]
    cams, radius = _rig(K, case.get("arc", 90.0), w, h)
    fr = _Frames(cams, seed)
    if kind == "views":
        n = case["views"]
        st = _State(case, cams, n_ref=case["n_ref"], frame_slots=n, max_batch=n, layered=int(case["layered"]),
                    pixel_weights=int(case["pixel_weights"]))
        if case["layered"]:
            model = fr.mm.clone()
            model[fr.fg] = 0
            model = model.round().clamp(0, 65534).int().to(torch.int16)
            torch.cuda.synchronize()
            for k in range(K):
                F.fvv_set_bg_depth(st.ctx, k, model[k].contiguous(), w * 2)
        for t in range(n):
            rgb, depth = fr.tick(case["layered"])
            torch.cuda.synchronize()
            _upload(st, t, rgb, depth)
            torch.cuda.synchronize()
        st.views = _swing(n, case["arc"], radius, case["vw"], case["vh"], fr.gen)
        st.ticks = list(range(n))
        shape = (case["vh"], case["vw"])
        st.out = [torch.zeros((*shape, 3), dtype=torch.uint8, device="cuda") for _ in range(n)]
        st.pitch = [case["vw"] * 3] * n
        st.depth, st.hole, st.aux = [], [], None
        if case["aux"]:
            st.depth = [torch.zeros(shape, dtype=torch.float32, device="cuda") for _ in range(n)]
            st.hole = [torch.zeros(shape, dtype=torch.uint8, device="cuda") for _ in range(n)]
            st.aux = [F.aux(d, m) for d, m in zip(st.depth, st.hole)]
        return st
    if kind == "tick":
        st = _State(case, cams, n_ref=case["n_ref"], jbf_radius=case["radius"], frame_slots=2)
        st.rgb, st.codes = fr.tick()
        if case["yuv"]:
            st.yuv = _yuv(st.codes)
            for k in range(K):
                F.fvv_set_depth_codec(st.ctx, k, F.fvv_depth_codec_default())
        st.tick = 0
        st.view = _swing(1, 90.0, radius, case["vw"], case["vh"], fr.gen)[0]
        st.out = torch.zeros((case["vh"], case["vw"], 3), dtype=torch.uint8, device="cuda")
        return st
    if kind == "codec":
        st = _State(case, cams)
        st.codes = fr.tick()[1]
        for k in range(K):
            F.fvv_set_depth_codec(st.ctx, k, F.fvv_depth_codec_default())
        st.yuv = torch.zeros((K, w * h * 3 // 2), dtype=torch.uint8, device="cuda")
        st.out = torch.zeros_like(st.codes)
        return st
    # serve: the viewer mix of the serving workload, 640x360 : 1280x720 : 1920x1080 = 2 : 1 : 1
    st = _State(case, cams, frame_slots=2)
    rgb, depth = fr.tick()
    torch.cuda.synchronize()
    _upload(st, 0, rgb, depth)
    torch.cuda.synchronize()
    sizes = [((640, 360), (1280, 720), (640, 360), (1920, 1080))[i % 4] for i in range(case["viewers"])]
    st.views = [_swing(1, 90.0, radius, *s, fr.gen)[0] for s in sizes]
    st.out = [torch.zeros((s[1], s[0], 3), dtype=torch.uint8, device="cuda") for s in sizes]
    F.fvv_serve_start(st.ctx, None)
    return st


# ---------------------------------------------------------------------------
# the refinement network's inputs: a plain synthesis, and weights
# ---------------------------------------------------------------------------
def _net_layers(case):
    w1, w2, w3 = case["w1"], case["w2"], case["w3"]
    return [(8, w1), (w1, w1), (w1, w2), (w2, w2), (w2, w3), (w3, w3), (w3 + w2, w2), (w2, w2), (w2 + w1, w1), (w1, w1)]


_SCALE = (1, 1, 4, 4, 16, 16, 4, 4, 1, 1)     # pixels per output of each layer


def _net_params(case, seed):
    """Flat weights in the library's order: W[cout][3][3][cin] and b per layer, then the 1x1 head."""
    g = torch.Generator().manual_seed(int(seed) + 77)
    parts = []
    for ci, co in _net_layers(case):
        parts += [torch.randn(co, 3, 3, ci, generator=g) * math.sqrt(2.0 / (9 * ci)), 0.01 * torch.randn(co, generator=g)]
    parts += [torch.randn(3, case["w1"], generator=g) * 0.02, 0.01 * torch.randn(3, generator=g)]
    return parts


def _net_inputs(case, seed):
    n, h, w = case["n"], case["h"], case["w"]
    g = torch.Generator().manual_seed(int(seed))
    dg = torch.Generator(device="cuda").manual_seed(int(seed))
    rgb, depth, target = [], [], []
    for i in range(n):
        c, z, _ = _raycast(_on_arc(-20.0 + 40.0 * float(torch.rand((), generator=g)), 1.5, 0.0, w, h), _scene(g))
        target.append(c)
        rgb.append(c + 12.0 * torch.randn(c.shape, device="cuda", generator=dg))
        depth.append(z * 1000.0 * (1 + 0.01 * torch.randn(z.shape, device="cuda", generator=dg)))
    top = torch.rand(n, h, w, 3, device="cuda", generator=dg).sort(-1, descending=True)[0]
    return {"rgb": torch.stack(rgb).clamp(0, 255).round().to(torch.uint8).contiguous(),
            "depth": torch.stack(depth).float().contiguous(),
            "hole": _gaps(n, h, w, dg).to(torch.uint8).contiguous(),
            "top3": (top / top.sum(-1, keepdim=True).clamp(min=1)).contiguous(),
            "target": torch.stack(target).clamp(0, 255).round().to(torch.uint8).contiguous()}


def _prepare_net(case, seed):
    st = _State(case, [_on_arc(0.0, 1.5, 0.0, 64, 64)], frame_slots=1, max_batch=1)
    F.fvv_refine_init(st.ctx, F.fvv_refine_default_cfg(widths=(case["w1"], case["w2"], case["w3"]), z_far=Z_FAR))
    F.fvv_refine_set(st.ctx, F.FVV_REFINE_PARAMS,
                     torch.cat([p.reshape(-1) for p in _net_params(case, seed)]).numpy())
    st.inp = _net_inputs(case, seed)
    st.batch = F.refine_batch(case["n"], case["h"], case["w"], st.inp["rgb"], st.inp["depth"], st.inp["hole"],
                              st.inp["top3"], st.inp["target"])
    torch.cuda.synchronize()
    if case["kind"] == "refine":
        st.out = torch.zeros((case["n"], case["h"], case["w"], 3), dtype=torch.float32, device="cuda")
        if case["e4m3"]:
            F.fvv_refine_quantize(st.ctx, calib=st.batch, stream=st.s)
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(st):
    c = st.case
    kind = c["kind"]
    if kind == "views":
        F.fvv_synthesize_batch(st.ctx, st.views, st.ticks, st.out, st.pitch, st.aux, st.s)
        return [st.out, st.depth, st.hole]
    if kind == "tick":
        K, H, W = st.codes.shape
        if c["yuv"]:
            F.fvv_upload_frames_yuv(st.ctx, st.rgb, H * W * 3, W * 3, st.yuv, H * W * 3 // 2, st.tick, st.s)
        else:
            _upload(st, st.tick, st.rgb, st.codes)
        st.tick += 1
        F.fvv_synthesize(st.ctx, st.view, st.out, c["vw"] * 3, None, st.s)
        return st.out
    if kind == "serve":
        t = [F.fvv_serve_submit(st.ctx, i, v, o, v.width * 3) for i, (v, o) in enumerate(zip(st.views, st.out))]
        for x in t:
            F.fvv_serve_poll(st.ctx, x)
        return st.out
    if kind == "codec":
        K, H, W = st.codes.shape
        p, d = st.yuv.data_ptr(), st.codes.data_ptr()
        fb = H * W * 3 // 2
        for k in range(K):
            y = p + k * fb
            F.fvv_depth_encode_yuv(st.ctx, k, d + k * H * W * 2, W * 2, y, W, y + H * W, y + H * W * 5 // 4, W // 2,
                                   st.s)
        F.fvv_depth_decode_yuv_frames(st.ctx, K, st.yuv, fb, st.out, H * W * 2, W * 2, st.s)
        return [st.yuv, st.out]
    if kind == "jbf":
        F.fvv_depth_jbf(st.rgb, c["w"] * 3, st.depth, c["w"] * 2, st.out, c["w"] * 2, c["w"], c["h"], st.opt, st.s)
        return st.out
    if kind == "refine":
        F.fvv_refine_forward(st.ctx, st.batch, None, st.out, st.s)
        return st.out
    # the loss and gradients of the batch (a learning rate of 0 leaves the weights as they are)
    loss = F.fvv_refine_train_step(st.ctx, st.batch, 0.0, st.s)
    return {"loss": torch.tensor(loss), "grads": F.fvv_refine_get(st.ctx, F.FVV_REFINE_GRADS)}


# ---------------------------------------------------------------------------
# what a pass cannot do without, and its result in 64 bits
# ---------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind in ("refine", "train"):
        px = case["n"] * case["h"] * case["w"]
        mac = sum(9 * a * b / d for (a, b), d in zip(_net_layers(case), _SCALE)) \
            + 3 * case["w1"]
        weights = sum(9 * a * b + b for a, b in _net_layers(case)) + 3 * case["w1"] + 3
        if kind == "refine":
            return {"bytes": px * (3 + 4 + 1 + 12 + 12) + 4 * weights, "flops": 2 * mac * px}
        return {"bytes": px * (3 + 4 + 1 + 12 + 3) + 8 * weights, "flops": 6 * mac * px}
    ns = case["w"] * case["h"]
    if kind == "jbf":
        return {"bytes": 7 * ns, "flops": 0.05 * ns * (2 * case["radius"] + 1) ** 2 * 6}
    K = case["cams"]
    if kind == "codec":                       # codes read, planes written; planes read, codes written
        return {"bytes": 2 * K * ns * 3.5, "flops": 0}
    if kind == "serve":
        nd = sum((640 * 360, 1280 * 720, 640 * 360, 1920 * 1080)[i % 4] for i in range(case["viewers"]))
        return {"bytes": 5 * K * ns + 3 * nd, "flops": _view_flops(K, ns, nd / case["viewers"]) * case["viewers"]}
    n, nd = case.get("views", 1), case["vw"] * case["vh"]
    na = case["n_ref"] or K
    if kind == "tick":                        # the tick read and written once, the view's references read, the view
        return {"bytes": K * ns * (3 + (1.5 if case["yuv"] else 2) + 6) + 5 * na * ns + 3 * nd,
                "flops": _view_flops(na, ns, nd)}
    per = 5 * na * ns + (8 if case["aux"] else 3) * nd + (2 * na * ns if case["layered"] else 0)
    return {"bytes": n * per, "flops": n * _view_flops(na, ns, nd)}


def _view_flops(na, ns, nd):
    """One projection (15 operations and 2 divisions) per source point and per pixel of each other reference,
    and a weighted sum of three channels."""
    return 19.0 * na * ns + 28.0 * (na - 1) * nd


def _net_exact(case, seed, grad):
    p = [x.double().cuda().requires_grad_(grad) for x in _net_params(case, seed)]
    i = _net_inputs(case, seed)
    rgb = i["rgb"].double() / 255.0
    x = torch.cat([rgb, (i["depth"].double() / Z_FAR)[..., None], i["hole"].double()[..., None], i["top3"].double()],
                  -1).permute(0, 3, 1, 2)
    f = torch.nn.functional

    def conv(k, t):
        return f.relu(f.conv2d(t, p[2 * k].permute(0, 3, 1, 2), p[2 * k + 1], padding=1))

    def up(t):
        return f.interpolate(t, scale_factor=2, mode="nearest")

    e1 = conv(1, conv(0, x))
    e2 = conv(3, conv(2, f.max_pool2d(e1, 2)))
    b = conv(5, conv(4, f.max_pool2d(e2, 2)))
    d2 = conv(7, conv(6, torch.cat([up(b), e2], 1)))
    d1 = conv(9, conv(8, torch.cat([up(d2), e1], 1)))
    res = f.conv2d(d1, p[20][:, :, None, None], p[21]).permute(0, 2, 3, 1)
    out = (rgb + res).clamp(0, 1)
    if not grad:
        return out.contiguous()
    loss = ((out - i["target"].double() / 255.0) ** 2).mean()
    loss.backward()
    return {"loss": loss.detach(), "grads": torch.cat([t.grad.reshape(-1) for t in p])}


def exact(case, seed):
    """The network's outputs in 64 bits.  Everything else returns bytes, whole
    codes, or the depth of a z-buffer's winners, which have no such value."""
    if case["kind"] not in ("refine", "train"):
        return None
    with torch.backends.cudnn.flags(enabled=False):
        if case["kind"] == "train":
            return _net_exact(case, seed, True)
        with torch.no_grad():
            return _net_exact(case, seed, False)
