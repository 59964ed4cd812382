"""The work this library is used for, as timed cases through its public entry points.

Every case is one call (or one training step) as a user's program makes it: frames through
Renderer.forward, training steps through render / render_views and autograd, batches of mixed
requests through BatchRenderer.forward, and the single stages (project, bin_and_sort,
composite_forward, composite_backward).  Sizes are those of the benchmark and the tests, and
draw() spreads them over the same ranges.  exact() restates the method in 64 bits with plain
torch: no tile list limits, no fused arithmetic, its own camera maps and its own gradients.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2412_12507_gb300 import render as ut
from paper_2412_12507_gb300 import synth

FIELDS = ("means", "log_scales", "quats", "opacity_logits", "sh")


def _case(name, kind, **kw):
    c = dict(kind=kind, scene="cube", n=1000, deg=3, model="pinhole", rs=False, w=64, h=64, tile_w=16, tile_h=16,
             colour=0, degree=2, kbuffer=0, views=1)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest frame: 1,000 Gaussians, 64x64 pinhole, no SH; a preview or a unit of a sweep
        _case("frame_pinhole64_1k", "frame", n=1000, deg=0),
        # an interactive fisheye frame: 100k Gaussians on a shell, 1280x720
        _case("frame_fisheye720_100k", "frame", scene="shell", n=100_000, model="fisheye", w=1280, h=720),
        # the headline frame: 1M Gaussians, 1920x1080 rolling-shutter fisheye
        _case("frame_rs1080_1m", "frame", n=1_000_000, model="fisheye", rs=True, w=1920, h=1080),
        # the headline training step on the same view: forward, L2 loss, gradients
        _case("train_rs1080_1m", "train", n=1_000_000, model="fisheye", rs=True, w=1920, h=1080),
        # a small training step on a ragged image: early training, thumbnails
        _case("train_ragged_20k", "train", n=20_000, deg=2, w=403, h=297),
        # the batched multi-view training step: 3M Gaussians, 8 views of three kinds
        _case("train_views8_3m", "views", scene="mixed", n=3_000_000, views=8, model="mixed", w=1920, h=1080),
        # the projection alone, on the headline view
        _case("project_rs1080_1m", "project", n=1_000_000, model="fisheye", rs=True, w=1920, h=1080),
        # the sorted key lists alone, with the 64-bit keys: 300k Gaussians, 1920x1080 pinhole
        _case("bin_keys_300k", "bin", scene="mixed", n=300_000, w=1920, h=1080),
        # compositing alone at 3840x2160 with the fast per-particle colours
        _case("composite_4k_200k", "composite", scene="mixed", n=200_000, w=3840, h=2160, colour=1),
        # compositing's gradients alone, other tile shape, 640x480
        _case("backward_32x8_200k", "backward", scene="mixed", n=200_000, model="fisheye", w=640, h=480, tile_w=32,
              tile_h=8),
        # a step with the per-ray sorted compositing (k = 16), forward and gradients
        _case("sorted_k16_100k", "sorted", scene="mixed", n=100_000, w=1280, h=720, kbuffer=16),
        # a server's batch: six requests over two scenes, mixed cameras and resolutions
        _case("batch6_mixed", "batch", scene="mixed", n=500_000, views=6, model="mixed", w=1280, h=720),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["frame", "frame", "train", "train", "views", "project", "bin", "composite", "backward",
                       "sorted", "batch"])
    n = _log(rng, 300, 1_500_000)
    w, h = _log(rng, 40, 2600), _log(rng, 40, 1500)
    c = _case(None, kind, scene=rng.choice(["cube", "shell", "mixed"]), n=n, deg=rng.randrange(4),
              model=rng.choice(["pinhole", "fisheye", "fisheye", "pinhole_radial"]), rs=rng.random() < 0.4, w=w, h=h)
    c["tile_w"], c["tile_h"] = rng.choice([(16, 16), (16, 16), (16, 16), (8, 8), (32, 8), (16, 32)])
    if kind in ("frame", "train", "composite", "backward"):
        c["colour"] = rng.choice([0, 0, 0, 1])
        if c["colour"] == 0:
            c["degree"] = rng.choice([2, 2, 2, 2, 3, 4])
    if kind == "sorted":
        c["kbuffer"] = rng.choice([1, 4, 8, 16])
        c["n"] = min(n, 200_000)
    if kind in ("views", "batch"):
        c["views"] = rng.randrange(2, 9)
        c["model"] = "mixed"
        c["n"] = min(n, 600_000)
        c["w"], c["h"] = min(w, 1600), min(h, 1100)
    return c


# ---------------------------------------------------------------- inputs

def _gen(seed, salt=0):
    return torch.Generator(device="cuda").manual_seed(1_000_003 * int(seed) + salt)


def _scene(kind, n, deg, seed):
    """The benchmark's recipes, drawn on the GPU: a box in front of the camera, a noisy shell, or
    70 % shell and 30 % uniform volume."""
    g = _gen(seed)
    nrm = lambda *s: torch.randn(s, generator=g, device="cuda")  # noqa: E731
    uni = lambda *s: torch.rand(s, generator=g, device="cuda")  # noqa: E731
    if kind == "cube":
        means = uni(n, 3) * 2 - 1 + torch.tensor([0.0, 0.0, 3.0], device="cuda")
        ls, lstd = -3.0 + 0.5 * nrm(n, 3), 1.0
    else:
        u = nrm(n, 3)
        means = u / u.norm(dim=1, keepdim=True) * (5.0 + 0.3 * nrm(n, 1))
        ls, lstd = (-4.0 + 0.7 * nrm(n, 3), 1.5) if kind == "shell" else (-4.5 + 0.8 * nrm(n, 3), 1.0)
        if kind == "mixed":
            vol = uni(n) < 0.3
            means = torch.where(vol[:, None], uni(n, 3) * 2 - 1, means)
    q = nrm(n, 4)
    q = q / q.norm(dim=1, keepdim=True)
    logits = lstd * nrm(n)
    sh = torch.empty((n, (deg + 1) ** 2, 3), device="cuda")
    sh[:, 0] = (uni(n, 3) - 0.5) * (2 * math.sqrt(math.pi))
    if deg:
        sh[:, 1:] = 0.1 * nrm(n, (deg + 1) ** 2 - 1, 3)
    return dict(means=means.contiguous(), log_scales=ls.contiguous(), quats=q.contiguous(),
                opacity_logits=logits.contiguous(), sh=sh.contiguous())


def _cam(case, seed):
    """One view: at the origin for the box and the shell, on the radius-4 orbit for the mix."""
    r = random.Random(7919 * int(seed) + 11)
    m, w, h = case["model"], case["w"], case["h"]
    k = (0.0, 0.0, 0.0, 0.0)
    if m == "fisheye":
        k = [r.uniform(-0.05, 0.05) for _ in range(4)]
    elif m == "pinhole_radial":
        k = [r.uniform(-0.1, 0.1), r.uniform(-0.05, 0.05), r.uniform(-0.02, 0.02), 0.0]
    f = w / math.pi if m == "fisheye" else (float(w) if case["scene"] == "cube" else 0.6 * w)
    q, t = (1, 0, 0, 0), (0, 0, 0)
    if case["scene"] == "mixed":
        az, el = r.uniform(0, 2 * math.pi), math.radians(r.uniform(-30, 30))
        q, t = synth.look_at_pose(4.0 * np.array([math.cos(el) * math.cos(az), -math.sin(el),
                                                  math.cos(el) * math.sin(az)]))
    kw = {}
    if case["rs"]:
        qe, te = synth.rs_end_pose(0.05, 2.0)
        if case["scene"] == "mixed":  # the same motion after the orbit pose: x_c' = R_e (R x + t) + t_e
            a, b = np.array(qe), np.array(q)
            qe = np.array([a[0] * b[0] - a[1:] @ b[1:], *(a[0] * b[1:] + b[0] * a[1:] + np.cross(a[1:], b[1:]))])
            te = _rot_np(a) @ np.array(t) + np.array(te)
        kw = dict(q_end=qe, t_end=te, rolling_shutter=1)
    return synth.camera(m, w, h, fx=f, fy=f, k=k, q=q, t=t, **kw)


def _rot_np(q):
    w, x, y, z = q
    return np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)],
                     [2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)],
                     [2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]])


def _cams(case, seed):
    """The views of a batch, cycling through pinhole, fisheye and rolling-shutter fisheye."""
    w, h = case["w"], case["h"]
    kinds = [("pinhole", w, h, 0), ("fisheye", (5 * w) // 6, (3 * h) // 2, 0),
             ("pinhole", w, h, 0), ("fisheye", w + w // 15, (7 * h) // 5, 1)]
    return synth.orbit_cameras(int(seed), [kinds[j % 4] for j in range(case["views"])])


def _opts(case):
    return synth.options(tile_w=case["tile_w"], tile_h=case["tile_h"], colour_mode=case["colour"],
                         kernel_degree=case["degree"], kbuffer=case["kbuffer"])


def _ut_scene(p, deg):
    return ut.Scene(*(p[k] for k in FIELDS), deg)


def _upstream(case, seed):
    g = _gen(seed, 77)
    return (torch.randn((3, case["h"], case["w"]), generator=g, device="cuda"),
            torch.randn((case["h"], case["w"]), generator=g, device="cuda"))


def _target(h, w, seed, salt=55):
    return torch.rand((3, h, w), generator=_gen(seed, salt), device="cuda")


def prepare(case, seed):
    kind, deg, opts = case["kind"], case["deg"], _opts(case)
    p = _scene(case["scene"], case["n"], deg, seed)
    s = dict(kind=kind, deg=deg, opts=opts)
    if kind in ("views", "batch"):
        s["cams"] = _cams(case, seed)
        if kind == "views":
            s["params"] = [p[k].requires_grad_(True) for k in FIELDS]
            s["targets"] = [_target(c["height"], c["width"], seed, 60 + j) for j, c in enumerate(s["cams"])]
            s["renderer"] = ut.BatchRenderer([], opts)
        else:  # two resident scenes, the second a quarter of the first
            p2 = _scene("mixed", max(case["n"] // 4, 1), deg, seed + 500)
            s["renderer"] = ut.BatchRenderer([_ut_scene(p, deg), _ut_scene(p2, deg)], opts)
            s["requests"] = [(j % 2, c) for j, c in enumerate(s["cams"])]
        return s
    cam = s["cam"] = _cam(case, seed)
    if kind == "train":
        s["params"] = [p[k].requires_grad_(True) for k in FIELDS]
        s["target"] = _target(case["h"], case["w"], seed)
        s["renderer"] = ut.Renderer(cam, opts)
        return s
    sc = s["scene"] = _ut_scene(p, deg)
    if kind in ("frame", "sorted"):
        s["renderer"] = ut.Renderer(cam, opts)
        if kind == "sorted":
            s["up"] = _upstream(case, seed)
        return s
    s["proj"] = ut.project(sc, cam, opts)
    if kind == "project":
        return s
    s["ws"] = ut.Workspace()
    if kind == "bin":  # buffers sized once, with room to spare, as a program that bins frame after frame does
        q = ut.project(_ut_scene(_scene(case["scene"], case["n"], 0, 0), 0), _cam(case, 0), opts)
        cap = 1024 + (3 * int(q.ntiles.sum(dtype=torch.int64).item())) // 2
        z = lambda *shape, t=torch.int32: torch.zeros(shape, dtype=t, device="cuda")  # noqa: E731
        s["bin"] = ut.Binning(z(cap), z(ut.tile_count(cam, opts), 2), z(1, t=torch.int64), z(cap, t=torch.int64), cap)
        return s
    K = int(s["proj"].ntiles.sum(dtype=torch.int64).item())
    s["bin"] = ut.bin_and_sort(s["proj"], cam, opts, max(K, 1), ws=s["ws"])
    s["cws"] = ut.Workspace()
    s["frame"] = ut.composite_forward(sc, cam, opts, s["proj"], s["bin"], ws=s["cws"])
    if kind == "backward":
        s["up"] = _upstream(case, seed)
    return s


def run(s):
    kind, opts = s["kind"], s["opts"]
    if kind == "frame":
        f = s["renderer"].forward(s["scene"])
        return f.rgb, f.alpha, f.t_final
    if kind == "train":
        rgb, alpha = ut.render(*s["params"], s["deg"], s["renderer"])
        loss = ((rgb - s["target"]) ** 2).mean()
        return (*torch.autograd.grad(loss, s["params"]), rgb.detach(), alpha.detach())
    if kind == "views":
        out = ut.render_views(*s["params"], s["deg"], s["cams"], s["renderer"])
        loss = sum(((rgb - t) ** 2).mean() for (rgb, _), t in zip(out, s["targets"]))
        return (*torch.autograd.grad(loss, s["params"]), *(t.detach() for pair in out for t in pair))
    if kind == "batch":
        return [t for f in s["renderer"].forward(s["requests"]) for t in (f.rgb, f.alpha)]
    if kind == "sorted":
        f = s["renderer"].forward(s["scene"])
        g = s["renderer"].backward(s["scene"], *s["up"])
        return (*(g[k] for k in FIELDS), f.rgb, f.alpha)
    if kind == "project":
        q = ut.project(s["scene"], s["cam"], opts, s["proj"])
        return q.mean2d, q.cov2d, q.depth, q.rect, q.ntiles
    if kind == "bin":
        b = ut.bin_and_sort(s["proj"], s["cam"], opts, s["bin"].capacity, want_keys=True, ws=s["ws"], out=s["bin"])
        return b.vals, b.ranges, b.k_dev, b.keys
    if kind == "composite":
        f = ut.composite_forward(s["scene"], s["cam"], opts, s["proj"], s["bin"], s["frame"], ws=s["cws"])
        return f.rgb, f.alpha, f.t_final
    g = ut.composite_backward(s["scene"], s["cam"], opts, s["proj"], s["bin"], s["frame"], *s["up"], s["cws"])
    return [g[k] for k in FIELDS]


def work(case):
    """Bytes: parameters read once, images (and for training the target or upstream, and the
    gradients) once.  Operations: the projection's sigma points and the pixels' rays and SH bases,
    which are known from the sizes; how many particles each pixel meets is known only from the data
    and is not counted."""
    kind, n, nsh = case["kind"], case["n"], (case["deg"] + 1) ** 2
    pix, parts = case["w"] * case["h"], n
    if kind in ("views", "batch"):
        c = _cams(case, 0)
        pix = sum(v["width"] * v["height"] for v in c)
        parts = n * case["views"]
        if kind == "batch":
            n = n + max(n // 4, 1)
            parts = sum((case["n"], max(case["n"] // 4, 1))[j % 2] for j in range(case["views"]))
    points = 7 * (4 if case["rs"] else 1) * (75 if case["model"] != "pinhole" else 30)
    scene, image = n * (44 + 12 * nsh), pix * 16
    if kind == "project":
        return dict(bytes=n * (44 + 36), flops=n * points)
    if kind == "bin":
        return dict(bytes=n * 16 + 8 * pix / (case["tile_w"] * case["tile_h"]), flops=0)
    if kind in ("frame", "batch"):
        return dict(bytes=scene + image, flops=parts * points + 120 * pix)
    if kind == "composite":
        return dict(bytes=scene + 8 * n + image, flops=120 * pix)
    if kind == "backward":
        return dict(bytes=2 * scene + 8 * n + 2 * image + 8 * pix, flops=120 * pix)
    return dict(bytes=2 * scene + image + 12 * pix, flops=parts * points + 240 * pix)  # training steps


# ---------------------------------------------------------------- the method in 64 bits

D = torch.float64


def _t(v):
    return torch.tensor(np.asarray(v, np.float64), dtype=D, device="cuda")


def _first_root(c, hi):
    """First zero of 1 + c1 u + c2 u^2 + ... on (0, hi], or None."""
    r = np.roots([*reversed(c), 1.0]) if any(c) else np.array([])
    r = [x.real for x in r if abs(x.imag) < 1e-9 and 0 < x.real <= hi]
    return min(r) if r else None


class _Cam64:
    def __init__(self, cam, opts):
        self.model, self.W, self.H = cam["model"], cam["width"], cam["height"]
        self.f, self.c = _t([cam["fx"], cam["fy"]]), _t([cam["cx"], cam["cy"]])
        self.k, self.near, self.rs, self.iters = cam["k"], cam["near_plane"], cam["rolling_shutter"], opts["rs_iters"]
        q0 = np.array(cam["q_start"]) / np.linalg.norm(cam["q_start"])
        q1 = np.array(cam["q_end"]) / np.linalg.norm(cam["q_end"])
        if q0 @ q1 < 0:
            q1 = -q1
        self.R0, self.T0 = _t(_rot_np(q0)), _t(cam["t_start"])
        self.dT = _t(cam["t_end"]) - self.T0 if self.rs else torch.zeros_like(self.T0)
        a, b = q1, np.array([q0[0], *-q0[1:]])
        v = a[0] * b[1:] + b[0] * a[1:] + np.cross(a[1:], b[1:])
        s = np.linalg.norm(v)
        self.phi = 2 * math.atan2(s, a[0] * b[0] - a[1:] @ b[1:]) if self.rs else 0.0
        self.ax = _t(v / s if s > 0 else [1.0, 0.0, 0.0])
        k = self.k
        if self.model == "fisheye":
            u = _first_root([3 * k[0], 5 * k[1], 7 * k[2], 9 * k[3]], math.pi ** 2 / 4)
            self.lim = math.sqrt(u) if u else math.pi / 2
        elif self.model == "pinhole_radial":
            u = _first_root([3 * k[0], 5 * k[1], 7 * k[2]], 100.0)
            self.lim = math.sqrt(u) if u else 1e6

    def curve(self, x):
        k, u = self.k, x * x
        if self.model == "fisheye":
            return x * (1 + u * (k[0] + u * (k[1] + u * (k[2] + u * k[3]))))
        return x * (1 + u * (k[0] + u * (k[1] + u * k[2])))

    def rotate(self, y, th):
        s, c = torch.sin(th)[..., None], torch.cos(th)[..., None]
        return y * c + torch.linalg.cross(self.ax.expand_as(y), y) * s + self.ax * ((y @ self.ax)[..., None] * (1 - c))

    def at(self, y, t):
        return (self.rotate(y, t * self.phi) if self.rs else y) + self.T0 + t[..., None] * self.dT

    def map(self, p):
        z = p[..., 2]
        if self.model == "fisheye":
            rho = p[..., :2].norm(dim=-1)
            th = torch.atan2(rho, z)
            s = torch.where(rho > 0, self.curve(th) / rho, 1 / z)
            return self.f * s[..., None] * p[..., :2] + self.c, (p.norm(dim=-1) > self.near) & (th <= self.lim)
        xn = p[..., :2] / z[..., None]
        if self.model == "pinhole":
            return self.f * xn + self.c, z > self.near
        r = xn.norm(dim=-1)
        return self.f * xn * (self.curve(r) / r.clamp_min(1e-300))[..., None] + self.c, (z > self.near) & (r <= self.lim)

    def project(self, x):
        y = x @ self.R0.T
        t = torch.full(y.shape[:-1], 0.5 if self.rs else 0.0, dtype=D, device="cuda")
        ok = torch.ones_like(t, dtype=torch.bool)
        for _ in range(self.iters if self.rs else 0):
            uv, v = self.map(self.at(y, t))
            ok &= v
            t = ((uv[..., 1] - 0.5) / (self.H - 1)).clamp(0, 1)
        uv, v = self.map(self.at(y, t))
        return uv, ok & v, t, y

    def rays(self):
        py, px = torch.meshgrid(torch.arange(self.H, device="cuda", dtype=D),
                                torch.arange(self.W, device="cuda", dtype=D), indexing="ij")
        m = (torch.stack([px, py], -1) + 0.5 - self.c) / self.f
        rd = m.norm(dim=-1)
        ok = torch.ones_like(rd, dtype=torch.bool)
        d = torch.cat([m, torch.ones_like(m[..., :1])], -1)
        if self.model != "pinhole":
            top = torch.tensor(self.lim, dtype=D)
            ok = rd <= float(self.curve(top))
            lo, hi = torch.zeros_like(rd), torch.full_like(rd, min(self.lim, 64.0 if self.model != "fisheye" else 2.0))
            for _ in range(70):
                mid = 0.5 * (lo + hi)
                up = self.curve(mid) > rd
                lo, hi = torch.where(up, lo, mid), torch.where(up, mid, hi)
            x, r = 0.5 * (lo + hi), rd.clamp_min(1e-300)
            if self.model == "fisheye":
                d = torch.cat([m * (torch.sin(x) / r)[..., None], torch.cos(x)[..., None]], -1)
            else:
                d[..., :2] = m * (x / r)[..., None]
        t = py / max(self.H - 1, 1) if self.rs else torch.zeros_like(py)
        T = self.T0 + t[..., None] * self.dT
        if self.rs:
            return self.rotate(-T, -t * self.phi) @ self.R0, self.rotate(d, -t * self.phi) @ self.R0, ok
        return -T @ self.R0, d @ self.R0, ok

    def centre(self, t):
        T = self.T0 + t[..., None] * self.dT
        return (self.rotate(-T, -t * self.phi) if self.rs else -T) @ self.R0


def _basis(d, deg):
    """Real spherical harmonics (Condon-Shortley phase) of unit directions."""
    x, y, z = d.unbind(-1)
    b = [torch.full_like(x, 0.5 / math.sqrt(math.pi))]
    n = lambda l, m: math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - m) / math.factorial(l + m)  # noqa: E731
                               * (2 if m else 1))
    if deg > 0:
        b += [-n(1, 1) * y, n(1, 0) * z, -n(1, 1) * x]
    if deg > 1:
        b += [6 * n(2, 2) * x * y, -3 * n(2, 1) * y * z, n(2, 0) * (3 * z * z - 1) / 2, -3 * n(2, 1) * x * z,
              3 * n(2, 2) * (x * x - y * y)]
    if deg > 2:
        b += [-15 * n(3, 3) * y * (3 * x * x - y * y), 30 * n(3, 2) * x * y * z, -1.5 * n(3, 1) * y * (5 * z * z - 1),
              n(3, 0) * z * (5 * z * z - 3) / 2, -1.5 * n(3, 1) * x * (5 * z * z - 1),
              15 * n(3, 2) * z * (x * x - y * y), -15 * n(3, 3) * x * (x * x - 3 * y * y)]
    return torch.stack(b, -1)


def _rot(q):
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)


def _project64(p, cam, opts):
    """v_mu, Sigma', depth and the pixel rectangle [x0, y0, x1, y1] (empty where culled)."""
    mu, R = p["means"], _rot(p["quats"])
    L = R * torch.exp(p["log_scales"])[:, None, :] * math.sqrt(3.0)  # (alpha, beta, kappa) = (1, 2, 0): lambda = 0
    v0, ok, t, y = cam.project(mu)
    pts = []
    for k in range(3):
        for sgn in (1.0, -1.0):
            v, o, _, _ = cam.project(mu + sgn * L[:, :, k])
            ok = ok & o
            pts.append(v)
    pts = torch.stack(pts)
    vm = pts.mean(0)
    dv = pts - vm
    d0 = v0 - vm
    cov = torch.stack([(dv[..., i] * dv[..., j]).sum(0) / 6 + 2 * d0[:, i] * d0[:, j] for i, j in
                       ((0, 0), (0, 1), (1, 1))], 1)
    sigma = torch.sigmoid(p["opacity_logits"])
    ok = ok & (sigma >= opts["alpha_min"])
    deg = opts["kernel_degree"]
    lam = 0.5 * 3.0 ** (2 - deg)
    reach = (torch.log(sigma / opts["alpha_min"]).clamp_min(0) / lam) ** (1.0 / deg)
    half = torch.clamp(reach, max=opts["extent_sigma"])[:, None] * torch.sqrt(cov[:, [0, 2]])
    size = _t([cam.W - 1, cam.H - 1])
    lo = torch.ceil(vm - half - 0.5).clamp_min(0)
    hi = torch.minimum(torch.floor(vm + half - 0.5), size)
    ok = ok & (lo <= hi).all(1)
    depth = cam.at(y, t).norm(dim=1)
    z = ok.to(D)
    rect = torch.cat([lo, hi], 1)
    rect[~ok] = _t([0, 0, -1, -1])
    return vm * z[:, None], cov * z[:, None], depth * z, rect, ok, t


def _render64(case, seed, grad=None, cam=None, p=None):
    """(rgb, alpha, t_final) of one view; with grad = f(rgb) -> (d_rgb, d_alpha), also the
    parameters' gradients.  Walks all 16x16 tiles' depth-sorted lists side by side, one list
    position per step."""
    opts = _opts(case)
    p = p or _scene(case["scene"], case["n"], case["deg"], seed)
    deg = case["deg"]
    p = {k: v.detach().to(D) for k, v in p.items()}
    cam = _Cam64(cam or _cam(case, seed), opts)
    with torch.no_grad():
        _, _, depth, rect, ok, tm = _project64(p, cam, opts)
    leaves = {k: v.requires_grad_(grad is not None) for k, v in p.items()}
    M_ = _rot(leaves["quats"]).transpose(1, 2) / torch.exp(leaves["log_scales"])[:, :, None]
    sig_ = torch.sigmoid(leaves["opacity_logits"])
    col_ = None
    if case["colour"] and deg:
        dirs = leaves["means"] - cam.centre(tm)
        b = _basis(dirs / dirs.norm(dim=1, keepdim=True), deg)
        col_ = (b[:, :, None] * leaves["sh"]).sum(1) + 0.5
    M, sig, mu, sh = M_.detach(), sig_.detach(), leaves["means"].detach(), leaves["sh"].detach()
    col = None if col_ is None else col_.detach()
    W, H, TX, TY = cam.W, cam.H, -(-cam.W // 16), -(-cam.H // 16)
    # per-tile lists in depth order
    ids = torch.nonzero(ok).squeeze(1)
    ids = ids[torch.sort(depth[ids], stable=True).indices]
    tr = torch.div(rect[ids], 16, rounding_mode="floor").long()
    tw = tr[:, 2] - tr[:, 0] + 1
    cnt = tw * (tr[:, 3] - tr[:, 1] + 1)
    owner = torch.repeat_interleave(torch.arange(ids.numel(), device="cuda"), cnt)
    local = torch.arange(owner.numel(), device="cuda") - torch.repeat_interleave(torch.cumsum(cnt, 0) - cnt, cnt)
    tile = (tr[owner, 1] + torch.div(local, tw[owner], rounding_mode="floor")) * TX + tr[owner, 0] + local % tw[owner]
    tile, order = torch.sort(tile, stable=True)
    lst = ids[owner[order]]
    del owner, local, order
    length = torch.bincount(tile, minlength=TX * TY)
    first = torch.cumsum(length, 0) - length
    # pixels per tile [tiles, 256]
    o, d, okp = cam.rays()
    pad = lambda v: torch.nn.functional.pad(v, (0, 0, 0, TX * 16 - W, 0, TY * 16 - H))  # noqa: E731

    def tiles(v):
        v = pad(v if v.dim() == 3 else v[..., None])
        return v.view(TY, 16, TX, 16, -1).permute(0, 2, 1, 3, 4).reshape(TX * TY, 256, -1)

    def image(v):
        return v.view(TY, TX, 16, 16, -1).permute(0, 2, 1, 3, 4).reshape(TY * 16, TX * 16, -1)[:H, :W]
    o, d, okp = tiles(o), tiles(d), tiles(okp.to(D))[..., 0] > 0
    d = torch.where(okp[..., None], d, _t([0, 0, 1]))
    o = torch.where(okp[..., None], o, _t([0, 0, 0]))
    yy, xx = torch.meshgrid(torch.arange(TY * 16, device="cuda", dtype=D), torch.arange(TX * 16, device="cuda", dtype=D),
                            indexing="ij")
    px = xx.view(TY, 16, TX, 16).permute(0, 2, 1, 3).reshape(TX * TY, 256)
    py = yy.view(TY, 16, TX, 16).permute(0, 2, 1, 3).reshape(TX * TY, 256)
    Y = None if col is not None else _basis(d / d.norm(dim=-1, keepdim=True), deg)
    kdeg, lam, K = opts["kernel_degree"], 0.5 * 3.0 ** (2 - opts["kernel_degree"]), opts["kbuffer"]
    amax, amin, tmin = opts["alpha_max"], opts["alpha_min"], opts["t_min"]

    def hit(g, a):
        """Pixels of tiles a that particle g (one per tile) reaches, and the response's parts."""
        Mg = M[g]
        og = torch.einsum("tij,tpj->tpi", Mg, o[a] - mu[g][:, None])
        dg = torch.einsum("tij,tpj->tpi", Mg, d[a])
        dd = (dg * dg).sum(-1)
        c = torch.linalg.cross(og, dg)
        w2 = (c * c).sum(-1) / dd
        resp = sig[g][:, None] * torch.exp(-lam * (w2 if kdeg == 2 else w2 ** (kdeg / 2)))
        r = rect[g]
        inside = (px[a] >= r[:, :1]) & (px[a] <= r[:, 2:3]) & (py[a] >= r[:, 1:2]) & (py[a] <= r[:, 3:4])
        c = col[g][:, None].expand(-1, 256, -1) if col is not None else 0.5 + Y[a] @ sh[g]
        return inside & (resp >= amin), resp, w2, og, dg, dd, c

    nt = TX * TY
    T, C = torch.ones((nt, 256), dtype=D, device="cuda"), torch.zeros((nt, 256, 3), dtype=D, device="cuda")
    done = ~okp
    steps = torch.zeros((nt, 256), dtype=torch.long, device="cuda")
    if K:
        tau_b = torch.full((nt, 256, K + 1), math.inf, dtype=D, device="cuda")
        val_b = torch.zeros((nt, 256, K + 1, 4), dtype=D, device="cuda")

    def blend(a, use, al, c):
        Tn = T[a] * (1 - al)
        stop = use & (Tn < tmin)
        use = use & ~stop
        C[a] += torch.where(use[..., None], c * (al * T[a])[..., None], 0.0)
        T[a] = torch.where(use, Tn, T[a])
        done[a] |= stop
        return use

    def walk(visit, alive):
        j = 0
        act = torch.nonzero(length > 0).squeeze(1)
        while act.numel():
            if j % 16 == 0:
                act = act[(length[act] > j) & alive(act, j)]
            a = act[length[act] > j]
            if not a.numel():
                break
            for b in a.split(4096):
                visit(lst[first[b] + j], b, j)
            j += 1

    def forward(g, a, j):
        h, resp, _, og, dg, dd, c = hit(g, a)
        h = h & ~done[a]
        al, c = resp.clamp(max=amax), c.clamp_min(0)
        if not K:
            use = blend(a, h, al, c)
            steps[a] = torch.where(use, j + 1, steps[a])
            return
        tau = -(og * dg).sum(-1) / dd
        tb, vb = tau_b[a], val_b[a]
        tb[..., K] = torch.where(h, tau, math.inf)
        vb[..., K, :] = torch.cat([al[..., None], c], -1)
        # the buffer's free entries hold tau = inf: fill one, or blend the closest of K + 1
        full = (tb[..., :K] < math.inf).all(-1)
        sel = torch.where(full, tb.argmin(-1), tb[..., :K].argmax(-1))
        v = vb.gather(-2, sel[..., None, None].expand(-1, -1, 1, 4))[..., 0, :]
        blend(a, h & full, v[..., 0], v[..., 1:])
        put = (h & (sel < K))[..., None]
        at = sel.clamp(max=K - 1)[..., None]
        tb[..., :K] = torch.where(put, tb[..., :K].scatter(-1, at, tb[..., K:]), tb[..., :K])
        vb[..., :K, :] = torch.where(put[..., None], vb[..., :K, :].scatter(-2, at[..., None].expand(-1, -1, 1, 4),
                                                                          vb[..., K:, :]), vb[..., :K, :])
        tau_b[a], val_b[a] = tb, vb

    with torch.no_grad():
        walk(forward, lambda a, j: ~done[a].all(1))
        if K:
            every = torch.arange(nt, device="cuda")
            for _ in range(K):
                t, sel = tau_b[..., :K].min(-1)
                v = val_b.gather(-2, sel[..., None, None].expand(-1, -1, 1, 4))[..., 0, :]
                blend(every, (t < math.inf) & ~done, v[..., 0], v[..., 1:])
                tau_b.scatter_(-1, sel[..., None], math.inf)
    rgb = image(C).permute(2, 0, 1).contiguous()
    tf = image(T)[..., 0].contiguous()
    out = (rgb, 1 - tf, tf)
    if grad is None:
        return out
    g_rgb, g_a = grad(rgb)
    g_rgb, g_a = tiles(g_rgb.to(D).permute(1, 2, 0)), tiles(g_a.to(D))[..., 0]
    n = mu.shape[0]
    acc = {k: torch.zeros(s, dtype=D, device="cuda") for k, s in
           dict(M=(n, 3, 3), mu=(n, 3), s=(n,), sh=sh.shape, col=(n, 3)).items()}
    gaT, left = g_a * T, C.clone()
    Tr = torch.ones_like(T)

    def backward(g, a, j):
        h, resp, w2, og, dg, dd, c = hit(g, a)
        h = h & (steps[a] > j)
        al, cc, t = resp.clamp(max=amax), c.clamp_min(0), Tr[a]
        w = al * t
        rem = left[a] - cc * w[..., None]
        dal = (g_rgb[a] * (cc * t[..., None] - rem / (1 - al)[..., None])).sum(-1) + gaT[a] / (1 - al)
        da = torch.where(h & (resp <= amax), dal, 0.0)
        wc = torch.where(h[..., None] & (c > 0), g_rgb[a] * w[..., None], 0.0)
        dw2 = da * resp * (-lam) * (1.0 if kdeg == 2 else 0.5 * kdeg * w2 ** (kdeg / 2 - 1))
        tau = -(og * dg).sum(-1) / dd
        v = 2 * dw2[..., None] * (og + tau[..., None] * dg)
        x = o[a] - mu[g][:, None] + tau[..., None] * d[a]
        acc["M"].index_add_(0, g, torch.einsum("tpi,tpj->tij", v, x))
        acc["mu"].index_add_(0, g, -torch.einsum("tij,tpi->tj", M[g], v))
        acc["s"].index_add_(0, g, (da * resp).sum(1) / sig[g])
        if col is None:
            acc["sh"].index_add_(0, g, torch.einsum("tpk,tpc->tkc", Y[a], wc))
        else:
            acc["col"].index_add_(0, g, wc.sum(1))
        left[a] = torch.where(h[..., None], rem, left[a])
        Tr[a] = torch.where(h, t * (1 - al), t)

    with torch.no_grad():
        last = steps.max(1).values
        walk(backward, lambda a, j: last[a] > j)
    roots, ups = [M_, sig_], [acc["M"], acc["s"]]
    if col_ is not None:
        roots, ups = roots + [col_], ups + [acc["col"]]
    g = torch.autograd.grad(roots, [leaves[k] for k in FIELDS], ups, allow_unused=True)
    g = {k: torch.zeros_like(leaves[k]) if v is None else v for k, v in zip(FIELDS, g)}
    g["means"] = g["means"] + acc["mu"]
    g["sh"] = g["sh"] + acc["sh"]
    return (*out, *(g[k] for k in FIELDS))


def exact(case, seed):
    kind = case["kind"]
    if kind == "bin":
        return None  # whole numbers
    if kind == "project":
        opts = _opts(case)
        p = {k: v.to(D) for k, v in _scene(case["scene"], case["n"], case["deg"], seed).items()}
        vm, cov, depth, _, _, _ = _project64(p, _Cam64(_cam(case, seed), opts), opts)
        return vm, cov, depth, None, None
    if kind in ("frame", "composite"):
        return _render64(case, seed)
    if kind == "sorted":
        rgb, alpha, _ = _render64(case, seed)
        return None, None, None, None, None, rgb, alpha
    if kind == "train":
        t = _target(case["h"], case["w"], seed).to(D)
        r = _render64(case, seed, lambda rgb: (2 * (rgb - t) / rgb.numel(), torch.zeros_like(rgb[0])))
        return (*r[3:], r[0], r[1])
    if kind == "backward":
        up = _upstream(case, seed)
        return list(_render64(case, seed, lambda rgb: up)[3:])
    if kind == "batch":
        p = [_scene(case["scene"], case["n"], case["deg"], seed),
             _scene("mixed", max(case["n"] // 4, 1), case["deg"], seed + 500)]
        return [t for j, c in enumerate(_cams(case, seed)) for t in _render64(case, seed, cam=c, p=p[j % 2])[:2]]
    return None  # several training views: the 64-bit walk takes minutes
