"""The work that a user has this framework do, as cases that can be timed.

Kinds of case, each through the public entry points of the Python package:

  stream   one simulation context, one frame per pass: push the frame, drain the
           previous frame's events into a device buffer, read back the denoised
           frame (adaptive mode: only flagged pixels are regressed).
  dense    the same in exhaustive mode (WLR+ESIM: every pixel regressed).
  batch    several sequences stepped together.
  wlr      the differentiable dense regression: one forward and one backward pass.
  wlr2     the second-order dense regression.
  quality  P/R/F and chamfer distance of an event set against a reference.
  render   one frame of the Monte Carlo renderer.

Inputs are drawn on the GPU from the seed: moving textured rectangles over a
smooth gradient or over a panning cell texture, with multiplicative
Gamma(spp, 1/spp) noise on the radiance, as a path tracer at `spp` samples
per pixel delivers it.
"""
from __future__ import annotations

import math
import os
from types import SimpleNamespace

import torch

import paper_2303_02608_gb300 as esim

LOG_EPS = 1e-3
RIDGE = 1e-4
REC709 = (0.2126, 0.7152, 0.0722)
FSCALE = (1.0, 1.0, 1.0, 8.0, 1.0, 1.0, 1.0)   # precision form: BF16 depth is stored as depth / 8
POOL = 8            # frames held by a streaming case, played forward and backward
TAUS = (5e-4, 1e-3, 2e-3, 5e-3, 1e-2)


# ------------------------------------------------------------------ the cases

def listed() -> list:
    return [
        # the smallest call: the 64x64 moving disc with a 7x7x3 window, one frame at a time
        # (an interactive preview; launches and host work are all of it)
        dict(name="stream_disc64", kind="stream", scene="disc", width=64, height=64, radius=3, frames=3,
             contrast=0.2, spp=4, precision="fp32", rgb=False),
        # the benchmark's headline workload: 1080p at 1 spp, 15x15x5 window, storage formats
        # (FP16 log brightness, BF16 features); about 2% of the pixels are regressed per frame
        dict(name="stream_1080p", kind="stream", scene="rects", width=1920, height=1080, radius=7, frames=5,
             contrast=0.1, spp=1, precision="mixed", rgb=True),
        # a panning camera over texture: every cell edge moves, a fifth of the pixels is regressed
        # per frame (the density that the paper reports for its scenes)
        dict(name="stream_pan1080p", kind="stream", scene="pan", width=1920, height=1080, radius=7, frames=5,
             contrast=0.1, spp=1, precision="mixed", rgb=True),
        # WLR+ESIM at 1080p: the reference that the adaptive simulator is judged against
        dict(name="dense_1080p", kind="dense", scene="rects", width=1920, height=1080, radius=7, frames=5,
             contrast=0.1, spp=1, precision="mixed", rgb=True),
        # WLR+ESIM in FP32 on a small odd-sized crop
        dict(name="dense_ragged", kind="dense", scene="rects", width=333, height=251, radius=5, frames=4,
             contrast=0.15, spp=4, precision="fp32", rgb=True),
        # many small sequences stepped together (a data-set generator): a few objects in each
        dict(name="batch_small", kind="batch", sizes="256x256,256x256,320x240,320x240", radius=7, frames=5,
             contrast=0.25, spp=4, precision="fp32", rgb=True),
        # the differentiation workload: 512x512x16, 7x7x3 window, gradients of radiance and bandwidths
        dict(name="wlr_512", kind="wlr", width=512, height=512, sequence=16, radius=3, frames=3, spp=2, rgb=True),
        # one step of a bandwidth fit on a small odd-sized luminance crop
        dict(name="wlr_ragged", kind="wlr", width=129, height=95, sequence=6, radius=4, frames=3, spp=4, rgb=False),
        # the second-order workload: 512x512x16, 7x7x3 window
        dict(name="wlr2_512", kind="wlr2", width=512, height=512, sequence=16, radius=3, frames=3, spp=2, rgb=True),
        # the second-order form on a small odd-sized luminance crop
        dict(name="wlr2_ragged", kind="wlr2", width=97, height=61, sequence=4, radius=3, frames=3, spp=4, rgb=False),
        # evaluation of one event set of the 1280x720x120 workload
        dict(name="quality_720p", kind="quality", width=1280, height=720, sequence=120, contrast=0.25),
        # one 1080p frame of the renderer at 4 spp with two interactions
        dict(name="render_1080p", kind="render", width=1920, height=1080, spp=4, bounces=2),
    ]


def _log_int(rng, lo: int, hi: int) -> int:
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng) -> dict:
    kind = rng.choice(("stream", "stream", "dense", "batch", "wlr", "wlr", "wlr2", "wlr2", "quality", "render"))
    rgb = rng.random() < 0.7
    if kind in ("stream", "dense"):
        w = _log_int(rng, 64, 1920)
        h = max(48, min(1080, int(w * rng.uniform(0.5, 1.0))))
        r, t = rng.choice(((3, 3), (5, 4), (7, 5), (7, 4)))
        return dict(kind=kind, scene=rng.choice(("rects", "pan")), width=w, height=h, radius=r, frames=t,
                    contrast=rng.choice((0.1, 0.15, 0.25)), spp=rng.choice((1, 2, 4)),
                    precision=rng.choice(("fp32", "mixed")), rgb=rgb)
    if kind == "batch":
        sizes = ["%dx%d" % (s, max(64, int(s * rng.uniform(0.6, 1.0)))) for s in
                 (_log_int(rng, 96, 320) for _ in range(rng.randint(2, 4)))]
        return dict(kind=kind, sizes=",".join(sizes), radius=rng.choice((5, 7)), frames=rng.choice((3, 5)),
                    contrast=rng.choice((0.25, 0.5)), spp=rng.choice((2, 4, 8)), precision="fp32", rgb=rgb)
    if kind == "wlr":
        w = _log_int(rng, 24, 512)
        r, t = rng.choice(((2, 2), (3, 3), (4, 3), (3, 1)))
        return dict(kind=kind, width=w, height=max(20, int(w * rng.uniform(0.6, 1.0))), sequence=rng.randint(t, 8),
                    radius=r, frames=t, spp=rng.choice((2, 4)), rgb=rgb)
    if kind == "wlr2":
        w = _log_int(rng, 24, 320)
        r, t = rng.choice(((2, 3), (3, 1), (3, 3), (4, 2), (5, 3), (7, 3)))
        if r > 3:
            w = min(w, 160)
        return dict(kind=kind, width=w, height=max(20, int(w * rng.uniform(0.6, 1.0))), sequence=rng.randint(1, 6),
                    radius=r, frames=t, spp=rng.choice((2, 4)), rgb=rgb)
    if kind == "quality":
        w = _log_int(rng, 96, 1280)
        return dict(kind=kind, width=w, height=max(64, int(w * rng.uniform(0.5, 0.8))), sequence=_log_int(rng, 6, 60),
                    contrast=rng.choice((0.25, 0.5, 1.0)))
    w = _log_int(rng, 80, 1920)
    return dict(kind=kind, width=w, height=max(60, min(1080, int(w * rng.uniform(0.5, 0.8)))),
                spp=rng.choice((1, 2, 4)), bounces=rng.choice((1, 2, 3)))


# --------------------------------------------------------------------- inputs

class _Scene:
    """Moving textured rectangles (or one disc) over a gradient or a panning
    cell texture; every number from the seed."""

    def __init__(self, kind: str, width: int, height: int, seed: int, spp: int, rgb: bool,
                 n_rects: int = 32):
        self.kind, self.W, self.H, self.spp, self.rgb = kind, width, height, spp, rgb
        self.dev = torch.device("cuda", torch.cuda.current_device())
        self.gen = torch.Generator(device=self.dev).manual_seed(seed)
        g = torch.Generator().manual_seed(seed)
        H, W = height, width
        self.rects = []
        for _ in range(0 if kind == "disc" else n_rects):
            v = torch.rand(9, generator=g).tolist()
            w, h = H / 16 + (H / 4 - H / 16) * v[0], H / 16 + (H / 4 - H / 16) * v[1]
            ang, spd = 2 * math.pi * v[4], 0.5 + 3.5 * v[5]
            nz = 0.7 + 0.3 * v[7]
            s, phi = math.sqrt(1 - nz * nz), 2 * math.pi * v[8]
            self.rects.append((1.0 + 9.0 * v[6], W * v[2] - w / 2, H * v[3] - h / 2, w, h, spd * math.cos(ang),
                               spd * math.sin(ang), (s * math.cos(phi), s * math.sin(phi), nz),
                               (0.05 + 0.9 * torch.rand(4, 4, 3, generator=g)).to(self.dev)))
        self.rects.sort(key=lambda r: -r[0])
        cells = torch.rand(6, H // 6 + 48, W // 6 + 80, generator=self.gen, device=self.dev)
        self.cells = cells
        self.start = (16.0 + 8.0 * float(torch.rand(1, generator=g)), 24.0 + 16.0 * float(torch.rand(1, generator=g)))

    @staticmethod
    def _shade(n):
        lx, ly, lz = (v / math.sqrt(0.3 ** 2 + 0.5 ** 2 + 1.0) for v in (0.3, 0.5, 1.0))
        return 0.3 + 0.7 * max(0.0, n[0] * lx + n[1] * ly + n[2] * lz)

    def clean(self, t: int) -> dict:
        H, W, dev = self.H, self.W, self.dev
        ys = torch.arange(H, device=dev, dtype=torch.float32) + 0.5
        xs = torch.arange(W, device=dev, dtype=torch.float32) + 0.5
        if self.kind == "pan":
            cy = torch.floor((ys + 0.7 * t) / 6.0).long()
            cx = torch.floor((xs + 1.7 * t) / 6.0).long()
            u = self.cells[:, cy[:, None], cx[None, :]]
            albedo = 0.1 + 0.8 * u[:3]
            depth = 10.0 * (0.8 + 0.4 * u[3])
            n = torch.stack([0.9 * (u[4] - 0.5), 0.9 * (u[5] - 0.5), torch.ones_like(u[4])])
            normal = n / n.norm(dim=0, keepdim=True)
            light = torch.tensor([0.3, 0.5, 1.0], device=dev).view(3, 1, 1) / math.sqrt(0.3 ** 2 + 0.5 ** 2 + 1.0)
            rad = albedo * (0.3 + 0.7 * (normal * light).sum(0).clamp_min(0.0))
        else:
            grad = (0.2 + 0.8 * (xs - 0.5) / max(W - 1, 1)).expand(H, W)
            albedo = grad.expand(3, H, W).clone()
            rad = albedo.clone()
            depth = torch.full((H, W), 5.0 if self.kind == "disc" else 10.0, device=dev)
            normal = torch.zeros(3, H, W, device=dev)
            normal[2] = 1.0
        if self.kind == "disc":
            # the disc bounces between the walls of the image
            span = W - 32.0
            p = (self.start[0] - 16.0 + 2.0 * t) % (2 * span)
            cx = 16.0 + (p if p <= span else 2 * span - p)
            m = (xs[None, :] - cx) ** 2 + (ys[:, None] - self.start[1]) ** 2 <= 144.0
            rad = torch.where(m, 2.0, rad)
            albedo = torch.where(m, 0.9, albedo)
            depth = torch.where(m, 2.0, depth)
        for z, x0, y0, w, h, vx, vy, n, alb in self.rects:
            X, Y = x0 + vx * t, y0 + vy * t
            ix0, ix1 = max(0, math.ceil(X - 0.5)), min(W, math.ceil(X + w - 0.5))
            iy0, iy1 = max(0, math.ceil(Y - 0.5)), min(H, math.ceil(Y + h - 0.5))
            if ix0 >= ix1 or iy0 >= iy1:
                continue
            cx = ((xs[ix0:ix1] - X) * (4.0 / w)).floor().long().clamp(0, 3)
            cy = ((ys[iy0:iy1] - Y) * (4.0 / h)).floor().long().clamp(0, 3)
            a = alb[cy[:, None], cx[None, :]].permute(2, 0, 1)
            albedo[:, iy0:iy1, ix0:ix1] = a
            rad[:, iy0:iy1, ix0:ix1] = a * self._shade(n)
            depth[iy0:iy1, ix0:ix1] = z
            normal[:, iy0:iy1, ix0:ix1] = torch.tensor(n, device=dev).view(3, 1, 1)
        if not self.rgb:
            rad = _luminance(rad)[None]
        return {"radiance": rad.contiguous(), "normal": normal, "albedo": albedo.contiguous(), "depth": depth}

    def frame(self, t: int) -> dict:
        f = self.clean(t)
        u = torch.rand((self.spp,) + tuple(f["radiance"].shape), generator=self.gen, device=self.dev)
        f["clean"] = f["radiance"]
        f["radiance"] = (f["clean"] * (-torch.log1p(-u)).mean(0)).contiguous()
        return f


def _luminance(rad):
    return rad[0] if rad.shape[0] == 1 else REC709[0] * rad[0] + REC709[1] * rad[1] + REC709[2] * rad[2]


def _planes(f: dict):
    return torch.cat([f["normal"], f["depth"][None], f["albedo"]], 0)


def _stored(f: dict) -> dict:
    """A frame in the precision form's storage formats."""
    fs = torch.tensor(FSCALE, device=f["depth"].device).view(7, 1, 1)
    return {"radiance": torch.log(_luminance(f["radiance"]) + LOG_EPS).half().contiguous(),
            "features": (_planes(f) / fs).to(torch.bfloat16).contiguous()}


def _seen(frame: dict):
    """(y, features) of a pushed frame in float64, as the simulator reads them."""
    if "features" in frame:
        fs = torch.tensor(FSCALE, dtype=torch.float64, device=frame["features"].device).view(7, 1, 1)
        return frame["radiance"].double(), frame["features"].double() * fs
    return torch.log(_luminance(frame["radiance"].double()) + LOG_EPS), _planes(frame).double()


def _push_order(k: int) -> int:
    """Pool index of the k-th frame of a stream: forward, then backward, and so on."""
    k %= 2 * (POOL - 1)
    return k if k < POOL else 2 * (POOL - 1) - k


def _stream_frames(case, seed):
    sc = _Scene(case["scene"], case["width"], case["height"], seed, case["spp"], case["rgb"])
    raw = [sc.frame(t) for t in range(POOL)]
    if case["precision"] == "mixed":
        frames = [_stored(f) for f in raw]
    else:
        frames = [{k: f[k] for k in ("radiance", "normal", "albedo", "depth")} for f in raw]
    return raw, frames


def _checkpoint(case, raw, frames):
    """The model state that a stream resumes from, at frame T - 1: the converged log
    brightness, and slopes fitted to it in a 7x7 window."""
    f, shown = raw[case["frames"] - 1], frames[case["frames"] - 1]
    x = _seen(shown)[1]
    y = torch.log(_luminance(f["clean"].double()) + LOG_EPS)
    theta = _fit([y], [x], torch.arange(y.numel(), device=y.device), 3)
    flat = x.reshape(7, -1).t()
    return {"l_last": y.reshape(-1).float(), "beta": theta[:, 3:].float().contiguous(),
            "xc": flat.float().contiguous()}


def _sim_config(case):
    extra = {}
    if case["precision"] == "mixed":
        extra = dict(radiance_fmt=esim.ESIM_AD_LOGLUMA_F16, feature_fmt=esim.ESIM_AD_FEAT_BF16,
                     precision=esim.ESIM_AD_MIXED, feature_scale=list(FSCALE))
    mode = esim.ESIM_AD_EXHAUSTIVE if case["kind"] == "dense" else esim.ESIM_AD_ADAPTIVE
    return lambda w, h: esim.SimConfig(width=w, height=h, radius=case["radius"], frames=case["frames"],
                                       contrast=case["contrast"], rgb=case["rgb"], mode=mode, log_eps=LOG_EPS,
                                       ridge=RIDGE, event_capacity=max(1 << 16, 8 * w * h), **extra)


def _batch_sizes(case):
    return [tuple(int(v) for v in s.split("x")) for s in case["sizes"].split(",")]


def _batch_frames(case, seed):
    """Per sequence a pool of frames; sequence i starts i frames into its own motion."""
    pools = []
    for i, (w, h) in enumerate(_batch_sizes(case)):
        sc = _Scene("rects", w, h, seed * 64 + i, case["spp"], case["rgb"], n_rects=4)
        raw = [sc.frame(t + i) for t in range(POOL)]
        pools.append([{k: f[k] for k in ("radiance", "normal", "albedo", "depth")} for f in raw])
    return pools


def _wlr_inputs(case, seed):
    sc = _Scene("rects", case["width"], case["height"], seed, case["spp"], case["rgb"])
    fr = [sc.frame(t) for t in range(case["sequence"])]
    b = 0.6 + 0.8 * torch.rand(7, generator=sc.gen, device=sc.dev)
    rad = torch.stack([f["radiance"] for f in fr])
    feat = torch.stack([_planes(f) for f in fr])
    target = torch.log(torch.stack([_luminance(f["clean"]) for f in fr]) + LOG_EPS)
    return rad, feat, b, target


def _quality_inputs(case, seed):
    """Signed event counts [F][H][W] of plain ESIM on the noise-free frames and on
    frames with the smooth residual noise that denoising leaves."""
    sc = _Scene("rects", case["width"], case["height"], seed, 1, False)
    F, H, W, C = case["sequence"], case["height"], case["width"], case["contrast"]
    out = [torch.zeros(F, H, W, dtype=torch.int32, device=sc.dev) for _ in range(2)]
    last = [None, None]
    for t in range(F):
        y = torch.log(sc.clean(t)["radiance"][0] + LOG_EPS)
        n = torch.randn(1, 1, H // 8 + 1, W // 8 + 1, generator=sc.gen, device=sc.dev)
        n = torch.nn.functional.interpolate(n, size=(H, W), mode="bilinear")[0, 0]
        for s, v in enumerate((y + 0.06 * n, y)):
            if t:
                d = v - last[s]
                k = torch.trunc(d / C)
                out[s][t] = k.int()
                last[s] = last[s] + k * C
            else:
                last[s] = v
    return out


def _render_scene(case, seed):
    j = [(seed * 2654435761 >> s) % 97 / 97.0 for s in (3, 11, 19)]
    # an open-fronted box with a ceiling light and three moving spheres
    spheres = [SimpleNamespace(center=(-0.45 + 0.1 * j[0], -0.65, -0.6), velocity=(0.012, 0.0, 0.004), radius=0.35,
                               albedo=(0.8, 0.8, 0.8)),
               SimpleNamespace(center=(0.45, -0.7, 0.1 - 0.2 * j[1]), velocity=(-0.008, 0.0, -0.006), radius=0.3,
                               albedo=(0.2, 0.4, 0.8)),
               SimpleNamespace(center=(0.0, 0.2 + 0.1 * j[2], -0.9), velocity=(0.0, -0.01, 0.0), radius=0.2,
                               albedo=(0.9, 0.6, 0.1))]
    return SimpleNamespace(width=case["width"], height=case["height"], spp=case["spp"], max_bounces=case["bounces"],
                           seed=seed & 0x7fffffff, cam_pos=(0.0, 0.0, 1.4), tan_half_fov_y=0.41421356,
                           box=(1.0, 1.0, 1.5),
                           wall_albedo=((0.63, 0.065, 0.05), (0.14, 0.45, 0.091), (0.725, 0.71, 0.68),
                                        (0.725, 0.71, 0.68), (0.725, 0.71, 0.68)),
                           back_albedo2=(0.2, 0.2, 0.25), checker=0.25, light=(-0.3, 0.3, -0.6, 0.0),
                           light_radiance=(17.0, 12.0, 4.0), eps=1e-4, spheres=spheres)


# ------------------------------------------------------------------- the pass

def prepare(case: dict, seed: int):
    kind, s = case["kind"], SimpleNamespace(kind=case["kind"])
    if kind in ("stream", "dense"):
        raw, s.frames = _stream_frames(case, seed)
        cfg = _sim_config(case)(case["width"], case["height"])
        s.sim = esim.Simulator(cfg)
        s.sink = torch.empty(12 * cfg.event_capacity, dtype=torch.uint8, device="cuda")
        for k in range(case["frames"]):      # the temporal window is full
            s.sim.push(s.frames[_push_order(k)])
        s.t = case["frames"]
        s.sim.events_into(s.sink)
        if kind == "stream":
            s.sim.set_state(**{k: v.cpu().numpy() for k, v in _checkpoint(case, raw, s.frames).items()})
    elif kind == "batch":
        # tile shape and lanes per pixel as a user's machine has them cached after the first tuning
        os.environ["ESIM_AD_BATCH_TILE"], os.environ["ESIM_AD_BATCH_LANES"] = "16", "8"
        s.pools = _batch_frames(case, seed)
        make = _sim_config(case)
        cfgs = [make(w, h) for w, h in _batch_sizes(case)]
        cfgs[0].event_capacity = sum(c.event_capacity for c in cfgs)
        s.n, s.cap = len(cfgs), cfgs[0].event_capacity
        s.batch = esim.Batch(cfgs)
        s.sink = torch.empty(12 * s.cap, dtype=torch.uint8, device="cuda")
        for k in range(case["frames"]):
            s.batch.step([p[_push_order(k)] for p in s.pools])
        s.t = case["frames"]
        s.batch.events_device(s.sink, s.cap)
    elif kind in ("wlr", "wlr2"):
        s.rad, s.feat, s.b, s.target = _wlr_inputs(case, seed)
        s.opts = dict(radius=case["radius"], frames=case["frames"], log_eps=LOG_EPS, ridge=RIDGE)
        if kind == "wlr":
            s.rad.requires_grad_(True)
            s.b.requires_grad_(True)
    elif kind == "quality":
        s.gen, s.ref = _quality_inputs(case, seed)
    else:
        s.scene, s.t = _render_scene(case, seed), 0
    return s


def run(s):
    if s.kind in ("stream", "dense"):
        s.sim.push(s.frames[_push_order(s.t)])
        s.sim.events_frame_into(s.t - 1, s.sink)     # the previous frame's events, beside this frame's kernels
        s.t += 1
        alpha, flags = s.sim.denoised()
        return {"alpha": alpha, "flags": flags}
    if s.kind == "batch":
        s.batch.step([p[_push_order(s.t)] for p in s.pools])
        s.t += 1
        s.batch.events_device(s.sink, s.cap)
        out = [s.batch.denoised(i) for i in range(s.n)]
        return {"alpha": [a for a, _ in out], "flags": [f for _, f in out]}
    if s.kind == "wlr":
        alpha = esim.wlr(s.rad, s.feat, s.b, **s.opts)
        loss = (alpha - s.target).square().mean()
        g_rad, g_b = torch.autograd.grad(loss, (s.rad, s.b))
        return {"alpha": alpha.detach(), "g_radiance": g_rad, "g_bandwidth": g_b}
    if s.kind == "wlr2":
        return {"alpha": esim.wlr2(s.rad, s.feat, s.b, **s.opts)}
    if s.kind == "quality":
        q = esim.quality(s.gen, s.ref, TAUS)
        return {k: q[k] for k in ("precision", "recall", "fscore", "chamfer", "n_gen", "n_ref")}
    s.t += 1
    return esim.render(s.scene, s.t - 1)


# ------------------------------------------------------------ its work, its values

def _pairs(w, h, sequence, r, t):
    """(centre, neighbour) pairs of a dense pass, windows clipped to the image and the sequence."""
    n1 = lambda n: sum(min(n - 1, c + r) - max(0, c - r) + 1 for c in range(n))   # noqa: E731
    return n1(w) * n1(h) * sum(min(t, f + 1) for f in range(sequence))


def work(case: dict) -> dict:
    """Bytes: inputs and outputs once.  Flops: per (centre, neighbour) pair the feature
    differences (14), the squared distance (18), the weight (1) and the weighted sums of the
    normal equations (11 + 110 + 19 first order); the solves."""
    kind = case["kind"]
    if kind in ("stream", "dense", "batch"):
        n = sum(w * h for w, h in _batch_sizes(case)) if kind == "batch" else case["width"] * case["height"]
        nb = (2 * case["radius"] + 1) ** 2 * case["frames"]
        pan = case.get("scene") == "pan"
        frac = 1.0 if kind == "dense" else 0.2 if pan else 0.02
        if kind == "stream" and case["scene"] == "disc":
            frac = 0.1
        px_in = 16 if case["precision"] == "mixed" else 28 + 4 * (3 if case["rgb"] else 1)
        ring = 16 if case["precision"] == "mixed" else 32
        return {"bytes": n * (px_in + ring + 32 + 5) + frac * n * 64, "flops": frac * n * (162.0 * nb + 1000)}
    if kind in ("wlr", "wlr2"):
        px = case["width"] * case["height"] * case["sequence"]
        c = 3 if case["rgb"] else 1
        pairs = _pairs(case["width"], case["height"], case["sequence"], case["radius"], case["frames"])
        if kind == "wlr":
            return {"bytes": px * 4 * (c + 7 + 1 + 1 + c), "flops": pairs * (162.0 + 94 + 52) + px * 900.0}
        # second order: 770 distinct weighted moments, and a 56 x 56 Cholesky factor
        return {"bytes": px * 4 * (c + 7 + 1), "flops": pairs * (33.0 + 101 + 2 * 770) + px * 63472.0}
    if kind == "quality":
        n = case["width"] * case["height"] * case["sequence"]
        return {"bytes": 8.0 * n, "flops": 4.0 * n}
    n = case["width"] * case["height"]
    return {"bytes": 44.0 * n, "flops": 400.0 * n * case["spp"] * case["bounces"]}


def _gather(y, x, pix, r):
    """Neighbourhoods of the pixels `pix` in one frame: y [P][K], feature differences are taken by
    the caller; out-of-image neighbours are masked.  Returns (y, x [P][K][7], mask, ox, oy, index)."""
    H, W = y.shape
    o = torch.arange(-r, r + 1, device=y.device)
    oy, ox = o.repeat_interleave(2 * r + 1), o.repeat(2 * r + 1)
    ny, nx = (pix // W)[:, None] + oy, (pix % W)[:, None] + ox
    ok = (ny >= 0) & (ny < H) & (nx >= 0) & (nx < W)
    i = ny.clamp(0, H - 1) * W + nx.clamp(0, W - 1)
    return y.reshape(-1)[i], x.reshape(7, -1).t()[i], ok, ox, oy, i


def _design(y, x, xc, pix, r, hb):
    """Design rows z = (1, offset / r, feature differences) [P][K][10], weights and y of one frame."""
    yn, xn, ok, ox, oy, i = _gather(y, x, pix, r)
    P, K = yn.shape
    z = torch.empty(P, K, 10, dtype=torch.float64, device=y.device)
    z[..., 0] = 1.0
    z[..., 1], z[..., 2] = ox.double() / r, oy.double() / r
    z[..., 3:] = xn - xc[:, None, :]
    w = torch.exp(-0.5 * (z[..., 1:] / hb).square().sum(-1)) * ok
    return z, w, yn, i


def _fit(ys, xs, pix, r, b=None, ridge=RIDGE):
    """First-order regression in float64: theta [P][10] of the pixels `pix` of the last frame over
    the frames given (theta[:, 0] is the denoised value)."""
    dev = ys[0].device
    hb = torch.ones(9, dtype=torch.float64, device=dev)
    if b is not None:
        hb[2:] = b.double()
    reg = torch.ones(10, dtype=torch.float64, device=dev)
    reg[0] = 0.0
    side = 2 * r + 1
    step = max(1, (1 << 22) // (side * side))
    out = []
    for p0 in range(0, pix.numel(), step):
        p = pix[p0:p0 + step]
        xc = xs[-1].reshape(7, -1).t()[p]
        A = torch.zeros(p.numel(), 10, 11, dtype=torch.float64, device=dev)
        for y, x in zip(ys, xs):
            z, w, yn, _ = _design(y, x, xc, p, r, hb)
            A += torch.bmm((z * w[..., None]).transpose(1, 2), torch.cat([z, yn[..., None]], -1))
        g = A[..., 10:].clone()
        A = A[..., :10].contiguous()
        A.diagonal(dim1=1, dim2=2).add_(ridge * A[:, 0, 0, None] * reg)
        out.append(torch.linalg.solve(A, g)[..., 0])
    return torch.cat(out)


def _exact_stream(case, seed):
    """The simulator's frames in float64: alpha of every pixel as the pass returns it."""
    raw, frames = _stream_frames(case, seed)
    T, r, C = case["frames"], case["radius"], case["contrast"]
    ys, xs = zip(*(_seen(f) for f in frames))
    every = torch.arange(ys[0].numel(), device=ys[0].device)
    order = [_push_order(k) for k in range(T + 1)]
    window = lambda k: order[max(0, k - T + 1):k + 1]   # noqa: E731
    if case["kind"] == "dense":
        th = _fit([ys[i] for i in window(T)], [xs[i] for i in window(T)], every, r)
        return {"alpha": th[:, 0].reshape(ys[0].shape), "flags": None}
    alpha = last = beta = xc = None
    for k in range(T + 1):
        x = xs[order[k]].reshape(7, -1).t()
        if k == T:   # resumed from the checkpoint
            st = _checkpoint(case, raw, frames)
            beta, xc, last = st["beta"].double(), st["xc"].double(), st["l_last"].double()
        pix = every if k == 0 else every[((beta * (xc - x)).sum(1)).square() >= C * C]
        th = _fit([ys[i] for i in window(k)], [xs[i] for i in window(k)], pix, r)
        if k == 0:
            alpha, last, beta, xc = th[:, 0].clone(), th[:, 0].clone(), th[:, 3:].clone(), x.clone()
            continue
        alpha[pix] = th[:, 0]
        d = th[:, 0] - last[pix]
        n = torch.trunc(d / C)
        last[pix] += n * C
        e = n != 0
        beta[pix[e]], xc[pix[e]] = th[e, 3:], x[pix[e]]
    return {"alpha": alpha.reshape(ys[0].shape), "flags": None}


def _exact_wlr(case, seed):
    """alpha and the gradients of the mean squared error in float64 from the normal equations of every centre."""
    rad, feat, b, target = _wlr_inputs(case, seed)
    F, C, H, W = rad.shape
    r, T, dev = case["radius"], case["frames"], rad.device
    lum = torch.stack([_luminance(f) for f in rad.double()])
    y, x, b64 = torch.log(lum + LOG_EPS), feat.double(), b.double()
    hb = torch.cat([torch.ones(2, dtype=torch.float64, device=dev), b64])
    reg = torch.ones(10, dtype=torch.float64, device=dev)
    reg[0] = 0.0
    alpha = torch.empty(F, H * W, dtype=torch.float64, device=dev)
    gy, gb = torch.zeros(F, H * W, dtype=torch.float64, device=dev), torch.zeros(7, dtype=torch.float64, device=dev)
    step = max(1, (1 << 22) // (2 * r + 1) ** 2)
    for f in range(F):
        for p0 in range(0, H * W, step):
            pix = torch.arange(p0, min(H * W, p0 + step), device=dev)
            xc = x[f].reshape(7, -1).t()[pix]
            A = torch.zeros(pix.numel(), 10, 11, dtype=torch.float64, device=dev)
            for tau in range(max(0, f - T + 1), f + 1):
                z, w, yn, _ = _design(y[tau], x[tau], xc, pix, r, hb)
                A += torch.bmm((z * w[..., None]).transpose(1, 2), torch.cat([z, yn[..., None]], -1))
            rhs = torch.zeros(pix.numel(), 10, 2, dtype=torch.float64, device=dev)
            rhs[..., 0], rhs[:, 0, 1] = A[..., 10], 1.0
            A = A[..., :10].contiguous()
            A.diagonal(dim1=1, dim2=2).add_(RIDGE * A[:, 0, 0, None] * reg)
            sol = torch.linalg.solve(A, rhs)
            theta, v = sol[..., 0], sol[..., 1]
            alpha[f, pix] = theta[:, 0]
            ga = 2.0 * (theta[:, 0] - target[f].reshape(-1)[pix].double()) / target.numel()
            pen = RIDGE * (v * theta * reg).sum(1)
            for tau in range(max(0, f - T + 1), f + 1):
                z, w, yn, i = _design(y[tau], x[tau], xc, pix, r, hb)
                vz, res = (z @ v[..., None])[..., 0], yn - (z @ theta[..., None])[..., 0]
                gy[tau].index_add_(0, i.reshape(-1), (ga[:, None] * w * vz).reshape(-1))
                c = ga[:, None] * (vz * res - pen[:, None]) * w
                gb += (c[..., None] * z[..., 3:].square()).sum((0, 1)) / b64 ** 3
    gl = (gy / (lum.reshape(F, -1) + LOG_EPS)).reshape(F, H, W)
    k = REC709 if C == 3 else (1.0,)
    return {"alpha": alpha.reshape(F, H, W), "g_radiance": torch.stack([c * gl for c in k], 1), "g_bandwidth": gb}


def _exact_wlr2(case, seed):
    rad, feat, b, _ = _wlr_inputs(case, seed)
    F, _, H, W = rad.shape
    r, T, dev = case["radius"], case["frames"], rad.device
    if F * H * W * (2 * r + 1) ** 2 * T > 200_000_000:
        return None
    y, x = torch.stack([torch.log(_luminance(f) + LOG_EPS) for f in rad.double()]), feat.double()
    hb = torch.cat([torch.ones(2, dtype=torch.float64, device=dev), b.double()])
    reg = torch.ones(55, dtype=torch.float64, device=dev)
    reg[0] = 0.0
    ia, ib = torch.triu_indices(9, 9, device=dev)
    alpha = torch.empty(F, H * W, dtype=torch.float64, device=dev)
    step = max(1, (1 << 20) // (2 * r + 1) ** 2)
    for f in range(F):
        for p0 in range(0, H * W, step):
            pix = torch.arange(p0, min(H * W, p0 + step), device=dev)
            xc = x[f].reshape(7, -1).t()[pix]
            A = torch.zeros(pix.numel(), 55, 56, dtype=torch.float64, device=dev)
            for tau in range(max(0, f - T + 1), f + 1):
                z, w, yn, _ = _design(y[tau], x[tau], xc, pix, r, hb)
                z = torch.cat([z, z[..., 1 + ia] * z[..., 1 + ib]], -1)
                A += torch.bmm((z * w[..., None]).transpose(1, 2), torch.cat([z, yn[..., None]], -1))
            g = A[..., 55:].clone()
            A = A[..., :55].contiguous()
            A.diagonal(dim1=1, dim2=2).add_(RIDGE * A[:, 0, 0, None] * reg)
            alpha[f, pix] = torch.linalg.solve(A, g)[:, 0, 0]
    return {"alpha": alpha.reshape(F, H, W)}


def _exact_quality(case, seed):
    gen, ref = _quality_inputs(case, seed)
    scale = torch.tensor([case["sequence"], case["height"], case["width"]], dtype=torch.float64, device=gen.device)
    pts = [[(c * pol > 0).nonzero() for pol in (1, -1)] for c in (gen, ref)]
    if max(a.shape[0] * float(b.shape[0]) for a, b in zip(*pts)) > 1e11:
        return None
    hits, sums, n = [[0] * len(TAUS), [0] * len(TAUS)], [0.0, 0.0], [int(gen.abs().sum()), int(ref.abs().sum())]
    for d, c in enumerate((gen, ref)):
        for q, o in zip(pts[d], pts[1 - d]):
            m = c[tuple(q.t())].abs().double()
            if q.shape[0] and not o.shape[0]:
                sums[d] = math.inf
                continue
            rows = max(1, (1 << 27) // max(1, o.shape[0]))
            for p0 in range(0, q.shape[0], rows):
                near = torch.cdist(q[p0:p0 + rows].double() / scale, o.double() / scale,
                                   compute_mode="donot_use_mm_for_euclid_dist").amin(1)
                mm = m[p0:p0 + rows]
                sums[d] += float((mm * near.square()).sum())
                for k, tau in enumerate(TAUS):
                    hits[d][k] += float(mm[near < tau].sum())
    P, R = ([h / max(1, n[d]) for h in hits[d]] for d in (0, 1))
    fs = [2 * p * q / (p + q) if p + q > 0 else 0.0 for p, q in zip(P, R)]
    as64 = lambda v: [torch.tensor(u, dtype=torch.float64) for u in v]   # noqa: E731
    return {"precision": as64(P), "recall": as64(R), "fscore": as64(fs),
            "chamfer": torch.tensor(sum(s / max(1, k) for s, k in zip(sums, n)), dtype=torch.float64),
            "n_gen": None, "n_ref": None}


def exact(case: dict, seed: int):
    if case["kind"] in ("stream", "dense"):
        return _exact_stream(case, seed)
    if case["kind"] == "wlr":
        return _exact_wlr(case, seed)
    if case["kind"] == "wlr2":
        return _exact_wlr2(case, seed)
    if case["kind"] == "quality":
        return _exact_quality(case, seed)
    # render: every value is defined by single-precision decisions (which surface a ray reaches);
    # batch: each sequence goes through its own frames as a stream does, seen above
    return None
