"""The work users have this library do, as timed cases.

Every case goes through the public binding (paper_2507_02674_gb300.glint and
render): whole frames (map update, then shading), shading under a static map
with the options that change its kernels, reflection probabilities, the
surrogate's training data, training and inference, and frames that start and
end in host memory.  Inputs are seeded scenes, maps and networks with the
distributions of the benchmark and the tests, made on the GPU.

exact() restates the computed quantities in float64 torch from their
definitions (radiance levels, weights, pyramid, filtered maps, microfacet
tables, quadrature, network, Adam).  Shaded images have no such value: their
counts are decided by comparing FP32 thresholds with hashed uniforms.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2507_02674_gb300 import glint, render
from paper_2507_02674_gb300.synth import EnvMap

S_MIN, S_MAX = 0.02 ** 0.5, 0.5 ** 0.5
LEVELS, SAMPLES, ELL = 8, 64, 1e-4
N_PAR = 64 * 64 + 64 + 64 * 64 + 64 + 64 * 16 + 16
EVAL = {"e1": glint.EVAL_E1, "e2": glint.EVAL_E2, "mlp": glint.EVAL_MLP, "e1a": glint.EVAL_E1_ANISO}
DRAW = {"dual": glint.DRAW_DUAL, "single": glint.DRAW_SINGLE, "single_old": glint.DRAW_SINGLE_OLD,
        "wang": glint.DRAW_WANG2020}
WFMT = {"f32": glint.WFMT_F32, "f16": glint.WFMT_F16, "unorm16": glint.WFMT_UNORM16, "unorm8": glint.WFMT_UNORM8}


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # a material preview: the 64 x 64 unit sphere under a 64 x 32 float map, launch- and latency-bound
        {"name": "preview_sphere", "kind": "frame", "scene": "sphere", "w": 64, "h": 64, "K": 4, "env_h": 32,
         "half": False, "out_w": 64},
        # the renderer's ordinary frame: dynamic 1024 x 512 map filtered anew, 1080p scene shaded
        {"name": "frame_1080p", "kind": "frame", "scene": "scene", "w": 1920, "h": 1080, "K": 8, "env_h": 512,
         "half": True, "out_w": 256},
        # the largest frame: 4K at grazing view (long footprints, background), 2048 x 1024 map, sixteen levels
        {"name": "frame_4k_grazing", "kind": "frame", "scene": "grazing", "w": 3840, "h": 2160, "K": 16,
         "env_h": 1024, "half": True, "out_w": 256},
        # a window of odd size under a static map with float16 weights, real counts, four levels
        {"name": "window_odd_k4", "kind": "shade", "scene": "scene", "w": 1283, "h": 717, "K": 4, "env_h": 512,
         "half": True, "out_w": 256, "wfmt": "f16", "count": "real", "evaluator": "e1", "draw": "dual", "grid": 0},
        # the anisotropic footprint grid: twelve samples a pixel
        {"name": "aniso_grid_720p", "kind": "shade", "scene": "scene", "w": 1280, "h": 720, "K": 8, "env_h": 512,
         "half": True, "out_w": 256, "wfmt": "f32", "count": "integer", "evaluator": "e1", "draw": "dual", "grid": 1},
        # the surrogate frame: inputs, BF16 network and draws of every pixel
        {"name": "surrogate_1080p", "kind": "shade", "scene": "scene", "w": 1920, "h": 1080, "K": 8, "env_h": 512,
         "half": True, "out_w": 256, "wfmt": "f32", "count": "integer", "evaluator": "mlp", "draw": "dual", "grid": 0},
        # the surrogate's training data: inputs and quadrature labels of a frame's pixels
        {"name": "labels_720p", "kind": "labels", "scene": "scene", "w": 1280, "h": 720, "K": 8, "env_h": 512,
         "half": True, "out_w": 256, "S": 32},
        # the surrogate's training: Adam steps on consecutive batches, forward and backward
        {"name": "train_8192", "kind": "train", "K": 8, "batch": 8192, "steps": 32, "rows": 262144},
        # evaluating a trained network on stored samples
        {"name": "network_rows", "kind": "forward", "K": 8, "rows": 1000003},
        # reflection probabilities of the multi-tap anisotropic evaluator
        {"name": "probs_aniso_1080p", "kind": "probs", "scene": "scene", "w": 1920, "h": 1080, "K": 8, "env_h": 512,
         "half": True, "out_w": 256, "evaluator": "e1a", "S": 16},
        # end to end: map texels and G-buffer in pinned host memory, image written back there
        {"name": "host_frame_1080p", "kind": "host", "scene": "scene", "w": 1920, "h": 1080, "K": 8, "env_h": 512,
         "half": True, "out_w": 256},
        # the serving loop: a burst of mixed frames from pinned host memory, both paths
        {"name": "serve_burst", "kind": "serve", "frames": 6, "w": 1920, "h": 1080, "K": 8, "env_h": 512,
         "half": True, "out_w": 256},
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["frame", "frame", "shade", "shade", "shade", "labels", "train", "forward", "probs", "host",
                       "serve"])
    env_h = 1 << rng.randint(5, 10)
    c = {"kind": kind, "K": rng.choice([2, 4, 8, 16]), "env_h": env_h, "half": rng.random() < 0.7,
         "out_w": rng.choice([64, 128, 256]), "scene": rng.choice(["scene", "scene", "grazing", "sphere"])}
    if kind == "frame":
        c.update(w=log(33, 3840), h=log(33, 2160))
    elif kind == "shade":
        c.update(w=log(65, 2560), h=log(65, 1440), wfmt=rng.choice(["f32", "f32", "f16", "unorm16", "unorm8"]),
                 count=rng.choice(["integer", "integer", "real"]), evaluator="e1", draw="dual", grid=0)
        what = rng.choice(["e1", "mlp", "e1a", "draw", "grid"])
        if what in ("mlp", "e1a"):
            c["evaluator"] = what
        elif what == "draw":
            c["draw"] = rng.choice(["single", "single_old", "wang"])
        elif what == "grid":
            c["grid"] = 1
        if what == "mlp":
            c["K"] = rng.choice([2, 4, 8])
    elif kind == "labels":
        c.update(w=log(64, 1280), h=log(64, 720), K=rng.choice([2, 4, 8]), S=rng.choice([8, 13, 16, 24, 32]))
    elif kind == "probs":
        c.update(w=log(64, 1280), h=log(64, 720), evaluator=rng.choice(["e1", "e1a", "e2"]),
                 S=rng.choice([7, 16, 24, 32]))
    elif kind == "train":
        c = {"kind": kind, "K": rng.choice([2, 4, 8]), "batch": log(500, 32768), "steps": rng.randint(8, 32),
             "rows": log(40000, 400000)}
    elif kind == "forward":
        c = {"kind": kind, "K": rng.choice([2, 4, 8]), "rows": log(100, 2000000)}
    elif kind == "host":
        c.update(w=log(64, 1920), h=log(64, 1080))
    else:
        c = {"kind": kind, "frames": rng.randint(2, 6), "w": log(160, 1920), "h": log(90, 1080),
             "K": rng.choice([2, 4, 8]), "env_h": env_h, "half": True, "out_w": c["out_w"]}
    return c


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 13)


def _rand(g, *shape, lo=0.0, hi=1.0):
    return lo + (hi - lo) * torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def _unit(v):
    return v / v.norm(dim=-1, keepdim=True)


def _env_map(env_h, half, seed):
    """Log-normal low-frequency sky (sigma 1.5) with four Gaussian suns of
    radiance 1e3 .. 1e5, RGBA16F stored / 16 or RGBA32F."""
    g = _gen(seed)
    H, W = env_h, 2 * env_h
    th = math.pi * (torch.arange(H, device="cuda", dtype=torch.float64) + 0.5) / H
    ph = 2 * math.pi * (torch.arange(W, device="cuda", dtype=torch.float64) + 0.5) / W
    st, ct = torch.sin(th)[:, None], torch.cos(th)[:, None]
    d = torch.stack([st * torch.cos(ph), ct.expand(H, W), st * torch.sin(ph)], -1)
    f = torch.zeros(H, W, device="cuda", dtype=torch.float64)
    k = _unit(_randn(g, 24, 3)) * _rand(g, 24, 1, lo=1.0, hi=6.0)
    shift, amp = _rand(g, 24, hi=2 * math.pi), _rand(g, 24, lo=0.5)
    for i in range(24):
        f += amp[i] * torch.cos(d @ k[i] + shift[i])
    f += 0.8 * d[..., 1]
    rad = torch.exp(1.5 * (f - f.mean()) / f.std())
    img = torch.stack([rad, rad * (0.95 + 0.05 * d[..., 1]), rad * (0.9 + 0.1 * d[..., 1]), torch.ones_like(rad)], -1)
    cy, sphi = _rand(g, 4, lo=-0.2, hi=0.95), _rand(g, 4, hi=2 * math.pi)
    bright, size = torch.exp(_rand(g, 4, lo=math.log(1e3), hi=math.log(1e5))), torch.deg2rad(_rand(g, 4, lo=1, hi=3))
    sy = torch.sqrt(1 - cy * cy)
    suns = torch.stack([sy * torch.cos(sphi), cy, sy * torch.sin(sphi)], -1)
    tint = torch.tensor([1.0, 0.96, 0.88], device="cuda", dtype=torch.float64)
    for i in range(4):
        a = torch.arccos((d @ suns[i]).clamp(-1, 1))
        img[..., :3] += (bright[i] * torch.exp(-0.5 * (a / size[i]) ** 2))[..., None] * tint
    scale = 4 if half else 0
    img[..., :3] /= 2.0 ** scale
    return img.to(torch.float16 if half else torch.float32).contiguous(), scale


def _sphere_uv(n, s=8.0):
    return (s * torch.atan2(n[..., 2], n[..., 0]) / (2 * math.pi), s * torch.arccos(n[..., 1].clamp(-1, 1)) / math.pi)


def _sphere_duv(n, dn, s=8.0):
    st = torch.sqrt((1 - n[..., 1] ** 2).clamp_min(1e-12))
    rxz = (n[..., 0] ** 2 + n[..., 2] ** 2).clamp_min(1e-12)
    return (s * (n[..., 0] * dn[..., 2] - n[..., 2] * dn[..., 0]) / rxz / (2 * math.pi), -s * dn[..., 1] / st / math.pi)


def _on_plane(p, n, o, d):
    """Where the rays o + t d meet the tangent planes (p, n), as seen from p."""
    nd = (n * d).sum(-1)
    nd = torch.where(nd.abs() > 1e-12, nd, torch.full_like(nd, 1e-12))
    return o + ((n * (p - o)).sum(-1) / nd)[..., None] * d - p


def _gbuffer(scene, w, h, seed):
    """(four planes, tangent), each (w h, 4) float32: the 64 x 64-style sphere
    seen head-on, or a ground plane with sixteen spheres seen from above
    ("scene": every pixel hits) or at 5 degrees ("grazing": half is sky)."""
    g = _gen(seed)
    f8 = dict(device="cuda", dtype=torch.float64)
    if scene == "sphere":
        y, x = torch.meshgrid(1 - (torch.arange(h, **f8) + 0.5) * (2.0 / h),
                              -1 + (torch.arange(w, **f8) + 0.5) * (2.0 / w), indexing="ij")
        r2 = x * x + y * y
        hit = r2 < 1
        p = n = torch.stack([x, y, torch.sqrt((1 - r2).clamp_min(0))], -1)
        d = torch.tensor([0.0, 0.0, -1.0], **f8).expand_as(p)
        o = p - 5 * d
        on_sphere, ns, dn = hit, n, 1.0
        px = _on_plane(p, n, o + torch.tensor([2.0 / w, 0, 0], **f8), d)
        py = _on_plane(p, n, o + torch.tensor([0, -2.0 / h, 0], **f8), d)
        u = v = du = dv = torch.zeros_like(r2)
        dudx = dvdx = dudy = dvdy = du
        ax = ay = _rand(g, 1, lo=0.1, hi=0.2).expand(h, w)
        N0, F0 = (10 ** _rand(g, 1, lo=3.5, hi=4.5)).expand(h, w), torch.full((h, w), 0.9, **f8)
    else:
        pitch, height, n_lo, n_hi = (35.0, 4.0, 3.0, 8.0) if scene == "scene" else (5.0, 1.0, 2.0, 9.0)
        radius = _rand(g, 16, lo=0.2)
        c = torch.stack([_rand(g, 16, lo=-6, hi=6), radius, _rand(g, 16, lo=-6, hi=6)], -1)
        pitch = math.radians(pitch)
        o = torch.tensor([0.0, height, 3.0 + height / math.tan(pitch)], **f8)
        fwd = torch.tensor([0.0, -math.sin(pitch), -math.cos(pitch)], **f8)
        right, up = torch.tensor([1.0, 0.0, 0.0], **f8), torch.tensor([0.0, math.cos(pitch), -math.sin(pitch)], **f8)
        half = math.tan(math.radians(30.0))

        def rays(dx, dy):
            sx = ((torch.arange(w, **f8) + dx + 0.5) * (2.0 / w) - 1) * half * w / h
            sy = (1 - (torch.arange(h, **f8) + dy + 0.5) * (2.0 / h)) * half
            return _unit(fwd + sx[None, :, None] * right + sy[:, None, None] * up)

        d = rays(0, 0)
        down = d[..., 1] < -1e-9
        t = torch.where(down, -height / d[..., 1].clamp_max(-1e-9), torch.inf)
        ball = torch.full((h, w), -1, device="cuda")
        for i in range(16):
            oc = o - c[i]
            b = d @ oc
            disc = b * b - (oc @ oc - radius[i] ** 2)
            ti = -b - torch.sqrt(disc.clamp_min(0))
            near = (disc > 0) & (ti > 1e-6) & (ti < t)
            t, ball = torch.where(near, ti, t), torch.where(near, i, ball)
        hit = torch.isfinite(t)
        p = o + torch.where(hit, t, 1.0)[..., None] * d
        on_sphere, k = ball >= 0, ball.clamp_min(0)
        ns = (p - c[k]) / radius[k][..., None]
        n = torch.where(on_sphere[..., None], ns, torch.tensor([0.0, 1.0, 0.0], **f8))
        px, py = _on_plane(p, n, o, rays(1, 0)), _on_plane(p, n, o, rays(0, 1))
        dn = 1.0 / radius[k][..., None]
        u, v, dudx, dvdx, dudy, dvdy = p[..., 0], p[..., 2], px[..., 0], px[..., 2], py[..., 0], py[..., 2]
        ax, ay = _rand(g, h, w, lo=0.03, hi=0.3), _rand(g, h, w, lo=0.03, hi=0.3)
        N0, F0 = 10 ** _rand(g, h, w, lo=n_lo, hi=n_hi), _rand(g, h, w, lo=0.5)
    su, sv = _sphere_uv(ns)
    sux, svx = _sphere_duv(ns, px * dn)
    suy, svy = _sphere_duv(ns, py * dn)

    def pick(a, b):
        return torch.where(on_sphere, a, b)

    sph = torch.atan2(ns[..., 2], ns[..., 0])
    zero = torch.zeros_like(sph)
    planes = [torch.cat([-d.expand(h, w, 3), torch.where(hit, N0, 0.0)[..., None]], -1),
              torch.cat([n, F0[..., None]], -1),
              torch.stack([pick(su, u), pick(sv, v), ax, ay], -1),
              torch.stack([pick(sux, dudx), pick(svx, dvdx), pick(suy, dudy), pick(svy, dvdy)], -1),
              torch.stack([pick(-torch.sin(sph), zero + 1), zero, pick(torch.cos(sph), zero), zero], -1)]
    planes = [q.reshape(-1, 4).to(torch.float32).contiguous() for q in planes]
    return planes[:4], planes[4]


def _network(K, seed):
    """Parameters of a network that corrects the prior as a trained one does:
    He-normal layers, small biases, a small output layer, unused columns 0."""
    g = _gen(seed)
    W1, W2, W3 = _randn(g, 64, 64) * (2 / 36) ** 0.5, _randn(g, 64, 64) * (2 / 64) ** 0.5, _randn(g, 64, 16) * 0.08
    b1, b2, b3 = _rand(g, 64, lo=-0.1, hi=0.1), _rand(g, 64, lo=-0.1, hi=0.1), _rand(g, 16, lo=-0.1, hi=0.1)
    W1[6 * K + 3:] = 0
    W3[:, K:] = 0
    b3[K:] = 0
    return torch.cat([v.reshape(-1) for v in (W1, b1, W2, b2, W3, b3)]).to(torch.float32).cpu().numpy()


def _samples(n, K, seed):
    """Stored training samples: inputs shaped like the surrogate's (a pixel's
    prior, the weights at five taps around it, three scalars), log-priors and
    target distributions."""
    g = _gen(seed)
    f4 = dict(generator=g, device="cuda")
    z = torch.randn(n, K, **f4) * 2
    prior = torch.softmax(z, -1)
    taps = [torch.softmax(z + 0.5 * torch.randn(n, K, **f4), -1) for _ in range(5)]
    x = torch.zeros(n, 64, device="cuda")
    x[:, :6 * K] = torch.cat([prior] + taps, -1)
    x[:, 6 * K:6 * K + 3] = 0.1 + 0.9 * torch.rand(n, 3, **f4)
    lp = torch.log(prior.clamp_min(1e-6))
    y = torch.softmax(z + 0.3 * (taps[1] - taps[3]) + 0.1 * torch.randn(n, K, **f4), -1)
    return x.to(torch.bfloat16).view(torch.int16).contiguous(), lp.contiguous(), y.contiguous()


def _adam_state(K, seed):
    """Moments and step count of a run in its middle."""
    g = _gen(seed + 101)
    v = 1e-7 * torch.exp(_randn(g, N_PAR))
    m = 0.1 * torch.sqrt(v) * _randn(g, N_PAR)
    used = torch.from_numpy(_used(K)).cuda()
    return [torch.where(used, a, 0.0).to(torch.float32).cpu().numpy() for a in (m, v)] + [1000]


def _used(K):
    u = np.ones(N_PAR, bool)
    u[N_PAR - 16 - 1024:N_PAR - 16].reshape(64, 16)[:, K:] = False
    u[N_PAR - 16 + K:] = False
    return u


@functools.lru_cache(maxsize=None)
def _ctx():
    return glint.Context(0)  # a program has one: the device and its tables


def _config(case):
    return glint.EnvConfig(K=case["K"], ell=ELL, levels=LEVELS, samples=SAMPLES, out_width=case["out_w"], s_min=S_MIN,
                           s_max=S_MAX, weight_format=WFMT[case.get("wfmt", "f32")])


def _frame(case, seed):
    tex, scale = _env_map(case["env_h"], case["half"], seed + 31)
    fr = render.Frame(_ctx(), EnvMap(np.zeros((case["env_h"], 2 * case["env_h"], 4),
                                              np.float16 if case["half"] else np.float32), scale), _config(case))
    fr.texels = tex
    return fr


def _pinned(t):
    return t.cpu().pin_memory()


def _serve_sizes(case):
    """The burst's frames: the given size and ones of 1/3 and 2/3 of its sides in turn."""
    return [(max(1, case["w"] * s // 3), max(1, case["h"] * s // 3)) for s in ([3, 1, 2, 1, 2, 1] * 4)[:case["frames"]]]


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "seed": seed & 0xFFFF}
    K = case["K"]
    if kind == "train":
        s["data"] = _samples(case["rows"], K, seed)
        s["net"] = glint.Mlp(_ctx(), K, case["batch"])
        s["net"].import_state(_network(K, seed), *_adam_state(K, seed))
        return s
    if kind == "forward":
        x, lp, _ = _samples(case["rows"], K, seed)
        s["data"] = x, lp
        s["net"] = glint.Mlp(_ctx(), K, 8192)
        s["net"].set_params(_network(K, seed))
        s["out"] = torch.empty(case["rows"], K, device="cuda")
        return s
    s["frame"] = _frame(case, seed)
    if kind == "serve":
        s["frame"].update_env()
        s["net"] = glint.Mlp(_ctx(), K, 8192)
        s["net"].set_params(_network(K, seed))
        s["reqs"] = []
        for i, (w, h) in enumerate(_serve_sizes(case)):
            planes, tan = _gbuffer("scene", w, h, seed + i)
            s["reqs"].append((w, h, [_pinned(p) for p in planes], _pinned(tan), torch.zeros(w * h, 4).pin_memory(),
                              glint.EVAL_MLP if i % 3 == 2 else glint.EVAL_E1))
        s["server"] = glint.Server(_ctx(), K, 1 << 30)
        s["env_id"] = s["server"].add_env(s["frame"].env, s["net"])
        return s
    s["planes"], s["tangent"] = _gbuffer(case["scene"], case["w"], case["h"], seed)
    npix = case["w"] * case["h"]
    if kind == "host":
        s["planes"] = [_pinned(p) for p in s["planes"]]
        s["texels"] = _pinned(s["frame"].texels)
        s["out"] = torch.zeros(npix, 4).pin_memory()
        s["pipe"] = glint.HostPipe(_ctx(), band_pixels=case["w"] * -(-case["h"] // 8), slots=8)
        return s
    if kind != "frame":
        s["frame"].update_env()  # a static map, filtered when it was loaded
    if kind == "shade" and case["evaluator"] == "mlp":
        s["net"] = glint.Mlp(_ctx(), K, 8192)
        s["net"].set_params(_network(K, seed))
    if kind in ("frame", "shade"):
        s["out"] = torch.empty(npix, 4, device="cuda")
    elif kind == "probs":
        s["out"] = torch.empty(npix, K, device="cuda")
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "train":
        net = s["net"]
        net.train(*s["data"], 0, c["batch"], c["steps"], 1e-3, 1e-4)
        return {"params": net.export(glint.MLP_PARAMS), "m": net.export(glint.MLP_ADAM_M),
                "v": net.export(glint.MLP_ADAM_V)}
    if kind == "forward":
        return s["net"].forward(*s["data"], out=s["out"])
    fr = s["frame"]
    if kind == "serve":
        srv, left = s["server"], set()
        for i, (w, h, planes, tan, out, ev) in enumerate(s["reqs"]):
            left.add(srv.submit(s["env_id"], planes, w, h, out, seed=s["seed"] + i, evaluator=ev, tangent=tan))
        while left:
            srv.tick()
            left -= {d[0] for d in srv.poll()}
        return [r[4] for r in s["reqs"]]
    w, h = c["w"], c["h"]
    if kind == "frame":
        fr.update_env()
        return fr.shade(s["planes"], w, h, out=s["out"], seed=s["seed"])
    if kind == "shade":
        count = glint.COUNT_REAL if c["count"] == "real" else glint.COUNT_INTEGER
        return fr.shade(s["planes"], w, h, out=s["out"], seed=s["seed"], count_mode=count, tangent=s["tangent"],
                        evaluator=EVAL[c["evaluator"]], mlp=s.get("net"), draw=DRAW[c["draw"]],
                        gamma=0.01 if c["draw"] == "wang" else 0.0, grid=c["grid"])
    if kind == "probs":
        return fr.probs(s["planes"], w, h, evaluator=EVAL[c["evaluator"]], e2_samples=c["S"], tangent=s["tangent"],
                        out=s["out"])
    if kind == "labels":
        x, lp, y = glint.mlp_generate(_ctx(), fr.env, s["planes"], w, h, s["tangent"], e2_samples=c["S"])
        return {"x": x, "lp": lp, "y": y}
    fr.texels.copy_(s["texels"], non_blocking=True)
    fr.update_env()
    s["pipe"].shade(fr.env, s["planes"], w, h, s["out"], seed=s["seed"], inputs_ready=True)
    return s["out"]


def work(case):
    """Bytes: inputs once and outputs once.  Flops: what a pixel's draws
    (about 60 a tree node and sample), look-ups, quadrature points and network
    rows take, and the map's weights, pyramid and filter samples."""
    kind, K = case["kind"], case["K"]
    net = 2 * (64 * 64 * 2 + 64 * K)
    if kind == "train":
        n = case["batch"] * case["steps"]
        return {"bytes": n * (128 + 8 * K) + 24 * N_PAR, "flops": 3 * net * n}
    if kind == "forward":
        n = case["rows"]
        return {"bytes": n * (128 + 8 * K), "flops": net * n}
    tex = 2 * case["env_h"] ** 2
    texels = tex * (8 if case["half"] else 16)
    filtered = sum(w * w // 2 for w in _widths(case["out_w"]))
    env = tex * 60 + filtered * SAMPLES * (80 + 16 * (3 + K))
    if kind == "serve":
        sizes = [w * h for w, h in _serve_sizes(case)]
        mlp = sum(sizes[2::3])
        return {"bytes": 80 * sum(sizes) + 16 * mlp, "flops": sum(sizes) * (300 + 360 * (K - 1)) + mlp * (net + 1000)}
    n = case["w"] * case["h"]
    if kind in ("frame", "host"):
        return {"bytes": 80 * n + texels, "flops": n * (300 + 360 * (K - 1)) + env}
    if kind == "shade":
        more = {"mlp": net + 1000, "e1a": 1000, "e1": 0}[case["evaluator"]]
        draws = 60 * (12 if case["grid"] else 6) * (1 if case["draw"] == "wang" else K - 1)
        return {"bytes": n * (80 + (16 if more else 0)), "flops": n * (300 + draws + more)}
    e2 = case["S"] ** 2 * (100 + 10 * K)
    if kind == "labels":
        return {"bytes": n * (64 + 128 + 8 * K), "flops": n * (e2 + 1300)}
    return {"bytes": n * ((48 if case["evaluator"] == "e1" else 64) + 4 * K),
            "flops": n * {"e1": 300, "e1a": 1300, "e2": e2}[case["evaluator"]]}


# ------------------------------------------------------------------ float64
def _widths(out_w):
    res = []
    for r in range(LEVELS):
        s = float(np.float32(S_MIN)) + (float(np.float32(S_MAX)) - float(np.float32(S_MIN))) * r / (LEVELS - 1)
        res.append(int(min(max(2.0 ** math.floor(math.log2(2 * math.pi / (s * s)) + 0.5), min(8, out_w)), out_w)))
    return res


def _pyramid64(tex, scale, K):
    """Levels of (h, 2h, 3 + K) channels: colour and fuzzy weights, each 2 x 2
    block averaged with its rows' solid angles."""
    rgb = tex.double()[..., :3] * 2.0 ** scale
    Y = (rgb @ torch.tensor([0.2126, 0.7152, 0.0722], device="cuda", dtype=torch.float64)).clamp_min(0)
    lo = max(float(Y.min()), float(np.float32(ELL)))
    hi = max(float(Y.max()), lo)
    L = torch.tensor([0.0] + [lo * (hi / lo) ** (k / (K - 1)) for k in range(1, K)], device="cuda", dtype=torch.float64)
    j = (torch.bucketize(Y, L, right=True) - 1).clamp(0, K - 2)
    t = ((Y - L[j]) / (L[j + 1] - L[j])).clamp(max=1.0)
    w = torch.zeros(*Y.shape, K, device="cuda", dtype=torch.float64)
    w.scatter_(-1, j[..., None], (1 - t)[..., None])
    w.scatter_(-1, j[..., None] + 1, t[..., None])
    lev = [torch.cat([rgb, w], -1)]
    while lev[-1].shape[0] > 1:
        a = lev[-1]
        H = a.shape[0]
        edge = torch.cos(math.pi * torch.arange(H + 1, device="cuda", dtype=torch.float64) / H)
        solid = (edge[:-1] - edge[1:])[:, None, None]
        b = (a * solid).unflatten(0, (H // 2, 2)).sum(1).unflatten(1, (H, 2)).mean(2)
        lev.append(b / solid.unflatten(0, (H // 2, 2)).sum(1))
    return lev


def _bilinear64(img, d):
    """Channels of an equirectangular image in directions d (wrap, clamp)."""
    H, W = img.shape[:2]
    x = torch.remainder(torch.atan2(d[..., 2], d[..., 0]), 2 * math.pi) * (W / (2 * math.pi)) - 0.5
    y = torch.arccos(d[..., 1].clamp(-1, 1)) * (H / math.pi) - 0.5
    x0, y0 = torch.floor(x), torch.floor(y)
    fx, fy = (x - x0)[..., None], (y - y0)[..., None]
    xa, ya, yb = x0.long() % W, y0.long().clamp(0, H - 1), (y0.long() + 1).clamp(0, H - 1)
    xb = (xa + 1) % W
    flat = img.reshape(H * W, -1)
    return ((1 - fy) * ((1 - fx) * flat[ya * W + xa] + fx * flat[ya * W + xb])
            + fy * ((1 - fx) * flat[yb * W + xa] + fx * flat[yb * W + xb]))


def _filtered64(pyr, out_w):
    """Filtered maps by importance sampling of the GGX lobe with Hammersley points."""
    H = pyr[0].shape[0]
    s_lo, s_hi = float(np.float32(S_MIN)), float(np.float32(S_MAX))
    j = np.arange(SAMPLES)
    u1 = (j + 0.5) / SAMPLES
    u2 = np.array([int(format(int(i), "032b")[::-1], 2) / 2.0 ** 32 for i in j])
    maps = []
    for r, W in enumerate(_widths(out_w)):
        a2 = (s_lo + (s_hi - s_lo) * r / (LEVELS - 1)) ** 4
        den = 1 - u1 + a2 * u1
        c2, s2, cos2 = (1 - u1) / den, a2 * u1 / den, (1 - u1 - a2 * u1) / den
        D = a2 / (math.pi * (s2 + a2 * c2) ** 2)
        lod = np.clip(0.5 * np.log2(4 / (SAMPLES * D) / (4 * math.pi / (2 * H * H))) - 0.5, 0, len(pyr) - 1)
        y, x = torch.meshgrid((torch.arange(W // 2, device="cuda", dtype=torch.float64) + 0.5) * (2 * math.pi / W),
                              (torch.arange(W, device="cuda", dtype=torch.float64) + 0.5) * (2 * math.pi / W),
                              indexing="ij")
        sy, cy, sx, cx = torch.sin(y), torch.cos(y), torch.sin(x), torch.cos(x)
        axis = torch.stack([sy * cx, cy, sy * sx], -1)
        e1, e2 = torch.stack([cy * cx, -sy, cy * sx], -1), torch.stack([-sx, torch.zeros_like(x), cx], -1)
        acc, n = 0.0, 0
        for k in range(SAMPLES):
            if not cos2[k] > 0:
                continue
            n += 1
            sin2, phi = 2 * math.sqrt(c2[k] * s2[k]), 2 * math.pi * u2[k]
            d = sin2 * math.cos(phi) * e1 + sin2 * math.sin(phi) * e2 + cos2[k] * axis
            m = int(lod[k])
            f = lod[k] - m
            acc = acc + (1 - f) * _bilinear64(pyr[m], d) + f * _bilinear64(pyr[min(m + 1, len(pyr) - 1)], d)
        maps.append(acc / max(n, 1))
    return maps


def _look64(maps, d, s):
    """Filtered channels at directions d and roughness parameters s = sqrt(alpha)."""
    s_lo, s_hi = float(np.float32(S_MIN)), float(np.float32(S_MAX))
    t = ((s - s_lo) * ((LEVELS - 1) / (s_hi - s_lo))).clamp(0, LEVELS - 1)
    res = torch.zeros(*s.shape, maps[0].shape[-1], device="cuda", dtype=torch.float64)
    for r in range(LEVELS):
        wr = (1 - (t - r).abs()).clamp_min(0)
        at = wr > 0
        if bool(at.any()):
            res[at] += wr[at][:, None] * _bilinear64(maps[r], d[at])
    return res


@functools.lru_cache(maxsize=None)
def _visible64(n=64, q=128):
    """Visible reflecting over total microfacet area V and 1 - V on the n x n
    table nodes over (mu_o, sqrt alpha)."""
    node = (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) / n
    mu, alpha = node[None, :, None], (node * node)[:, None, None]
    s = (torch.arange(q * q, device="cuda", dtype=torch.float64) + 0.5) / (q * q)
    V = []
    for j in range(n):
        a = alpha[j]
        w = torch.sqrt(a * a + (1 - a * a) * s * s)
        cot = (s * s - a * a * (1 - s * s)) / (2 * s * a * torch.sqrt(1 - s * s))
        m = torch.arccos((-(mu[0] / torch.sqrt(1 - mu[0] ** 2)) * cot).clamp(-1, 1))
        V.append((w * m).sum(-1) / (math.pi * w.sum(-1)))
    V = torch.stack(V)
    return torch.stack([V, 1 - V], -1)


def _table64(mu, s):
    t = _visible64()
    n = t.shape[0]
    x, y = (mu * n - 0.5).clamp(0, n - 1), (s * n - 0.5).clamp(0, n - 1)
    x0, y0 = torch.floor(x).long(), torch.floor(y).long()
    x1, y1 = (x0 + 1).clamp_max(n - 1), (y0 + 1).clamp_max(n - 1)
    fx, fy = (x - x0)[:, None], (y - y0)[:, None]
    return (1 - fy) * ((1 - fx) * t[y0, x0] + fx * t[y0, x1]) + fy * ((1 - fx) * t[y1, x0] + fx * t[y1, x1])


def _geometry64(planes, tan):
    wo, n = planes[0][:, :3].double(), planes[1][:, :3].double()
    mu = (wo * n).sum(-1)
    t = tan[:, :3].double()
    t = _unit(t - (t * n).sum(-1, keepdim=True) * n)
    return wo, n, mu, t, torch.linalg.cross(n, t), planes[2][:, 2].double(), planes[2][:, 3].double()


def _probs64(case, planes, tan, maps):
    """E1's and (evaluator "e1a") the multi-tap anisotropic E1's p_k."""
    wo, n, mu, t, b, ax, ay = _geometry64(planes, tan)
    r = 2 * mu[:, None] * n - wo
    s = torch.sqrt(torch.sqrt(ax * ay))
    VU = _table64(mu.clamp(1e-4, 1), s)
    if case.get("evaluator") == "e1a":
        jt = -2 * ((wo * t).sum(-1, keepdim=True) * n + mu[:, None] * t)
        jb = -2 * ((wo * b).sum(-1, keepdim=True) * n + mu[:, None] * b)
        nt, nb = jt.norm(dim=-1), jb.norm(dim=-1)
        Lt, Lb = nt * ax, nb * ay
        u = torch.where((Lt >= Lb)[:, None], jt / nt[:, None], jb / nb[:, None])
        lo, hi = torch.minimum(Lt, Lb), torch.maximum(Lt, Lb)
        sig = torch.sqrt(0.4 * (hi * hi - lo * lo))
        s1 = torch.sqrt((0.5 * lo).clamp(1e-4, 1))
        xj, wj = np.polynomial.hermite_e.hermegauss(5)
        W = sum(w / math.sqrt(2 * math.pi) * _look64(maps, _unit(r + (x * sig)[:, None] * u), s1)
                for x, w in zip(xj, wj))[:, 3:]
    else:
        W = _look64(maps, r, s)[:, 3:]
    p = VU[:, :1] * W
    p[:, :1] += VU[:, 1:]
    return p


def _quadrature64(S, planes, tan, pyr):
    """E2's p_k: an S x S rule over the anisotropic slope distribution."""
    H = pyr[0].shape[0]
    K = pyr[0].shape[-1] - 3
    # the pyramid level is chosen by an exact FP32 comparison
    lx = torch.minimum(planes[2][:, 2], planes[2][:, 3]) * np.float32(4.0 / S).item()
    m = torch.zeros(lx.shape, dtype=torch.long, device="cuda")
    for k in range(len(pyr)):
        m = torch.where(float(H >> k) * lx >= np.float32(math.pi).item(), k, m)
    out = torch.empty(lx.shape[0], K, device="cuda", dtype=torch.float64)
    sv = (torch.arange(S, device="cuda", dtype=torch.float64) + 0.5) / S
    rr = (torch.sqrt(1 - sv * sv) / sv).repeat_interleave(S)
    ph = (2 * math.pi * sv).repeat(S)
    sv = sv.repeat_interleave(S)
    cp, sp = torch.cos(ph), torch.sin(ph)
    for level in range(len(pyr)):
        rows = torch.nonzero(m == level)[:, 0]
        for idx in rows.split(max(1, (1 << 23) // (S * S))):
            wo, n, mu, t, b, ax, ay = (v[:, None] for v in _geometry64([p[idx] for p in planes], tan[idx]))
            sx, sy = ax * (rr * cp), ay * (rr * sp)
            wgt = 2 * torch.sqrt(sv * sv + ((ax * cp) ** 2 + (ay * sp) ** 2) * (1 - sv * sv))
            h = n - sx[..., None] * t - sy[..., None] * b
            h2, oh = (1 + sx * sx + sy * sy), (h * wo).sum(-1)
            d = (2 * oh / h2)[..., None] * h - wo
            ok = 2 * oh - mu * h2 > 0
            w = _bilinear64(pyr[level][..., 3:], _unit(d))
            p = ((wgt * ok)[..., None] * w).sum(1)
            p[:, 0] += (wgt * ~ok).sum(1)
            out[idx] = p / wgt.sum(1, keepdim=True)
    return out


def _bf16(t):
    return t.to(torch.float32).to(torch.bfloat16).double()


def _split(p):
    W1, b1, W2, b2, W3, b3 = p.split([4096, 64, 4096, 64, 1024, 16])
    return W1.view(64, 64), b1, W2.view(64, 64), b2, W3.view(64, 16), b3


def _net64(p, x, lp, K):
    W1, b1, W2, b2, W3, b3 = _split(p)
    h1 = _bf16((x @ _bf16(W1) + b1).clamp_min(0))
    h2 = _bf16((h1 @ _bf16(W2) + b2).clamp_min(0))
    return h1, h2, torch.softmax((h2 @ _bf16(W3) + b3)[:, :K] + lp, -1)


def _train64(case, seed):
    """The Adam steps in float64, rounding to BF16 where the definition does:
    inputs, weights, activations and backpropagated signals."""
    K, B, steps = case["K"], case["batch"], case["steps"]
    x, lp, y = _samples(case["rows"], K, seed)
    x, lp, y = x.view(torch.bfloat16).double(), lp.double(), y.double()
    p = torch.from_numpy(_network(K, seed)).cuda().double()
    m, v, t = _adam_state(K, seed)
    m, v = torch.from_numpy(m).cuda().double(), torch.from_numpy(v).cuda().double()
    used = torch.from_numpy(_used(K)).cuda()
    lr_max, lr_min = np.float32(1e-3).item(), np.float32(1e-4).item()
    for i in range(steps):
        at = (i * B + torch.arange(B, device="cuda")) % case["rows"]
        xb, yb = x[at], y[at]
        W1, b1, W2, b2, W3, b3 = _split(p)
        h1, h2, q = _net64(p, xb, lp[at], K)
        d = q - yb
        z3 = torch.zeros(B, 16, device="cuda", dtype=torch.float64)
        z3[:, :K] = 2 * q * (d - (q * d).sum(-1, keepdim=True)) / B
        z3 = _bf16(z3)
        z2 = _bf16((z3 @ _bf16(W3).T) * (h2 > 0))
        z1 = _bf16((z2 @ _bf16(W2).T) * (h1 > 0))
        g = torch.cat([(xb.T @ z1).reshape(-1), z1.sum(0), (h1.T @ z2).reshape(-1), z2.sum(0),
                       (h2.T @ z3).reshape(-1), z3.sum(0)])
        g = torch.where(used, g, 0.0)
        t += 1
        m = torch.where(used, 0.9 * m + 0.1 * g, m)
        v = torch.where(used, 0.999 * v + 0.001 * g * g, v)
        lr = max(lr_max * 0.5 * (1 + math.cos(math.pi * i / steps)), lr_min)
        step = lr * (m / (1 - 0.9 ** t)) / (torch.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
        p = torch.where(used, p - step, p)
    return {"params": p, "m": m, "v": v}


def exact(case, seed):
    kind, K = case["kind"], case["K"]
    if kind == "train":
        return _train64(case, seed)
    if kind == "forward":
        x, lp, _ = _samples(case["rows"], K, seed)
        p = torch.from_numpy(_network(K, seed)).cuda().double()
        return torch.cat([_net64(p, a.view(torch.bfloat16).double(), b.double(), K)[2]
                          for a, b in zip(x.split(1 << 18), lp.split(1 << 18))])
    if kind not in ("labels", "probs"):
        return None  # images: the counts have no value apart from FP32 thresholds
    planes, tan = _gbuffer(case["scene"], case["w"], case["h"], seed)
    tex, scale = _env_map(case["env_h"], case["half"], seed + 31)
    pyr = _pyramid64(tex, scale, K)
    fg = planes[0][:, 3] > 0
    at = torch.nonzero(fg)[:, 0]
    planes, tan = [p[at] for p in planes], tan[at]

    def scatter(p):
        out = torch.zeros(fg.shape[0], K, device="cuda", dtype=torch.float64)
        out[at] = p
        return out

    if kind == "probs":
        if case["evaluator"] == "e2":
            return scatter(_quadrature64(case["S"], planes, tan, pyr))
        return scatter(_probs64(case, planes, tan, _filtered64(pyr, case["out_w"])))
    prior = _probs64(case, planes, tan, _filtered64(pyr, case["out_w"]))
    return {"x": None, "lp": scatter(torch.log(prior.clamp_min(1e-6))),
            "y": scatter(_quadrature64(case["S"], planes, tan, pyr))}
