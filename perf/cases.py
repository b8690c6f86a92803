"""The workloads this library is timed on: what a renderer, an inverse renderer and an
asset pipeline call, through the public entry points (api, autograd.shade, TextureFit).

Frames are ray-cast here, on the device, from seeded cameras: an orbit around a sphere on a
ground plane, views of a quad, tilted planes in Voronoi regions of the screen.  Textures hold
one smooth cosine-power lobe per bucket.  `exact` is the same lookup in FP64 with plain torch.
"""
import math
import random

import numpy as np
import torch

from paper_2301_01719_gb300 import api, autograd, fit

DEV = "cuda"
STORAGES = ("f32", "f16", "bf16", "e4m3")
FILTERS = ("nearest", "angular_bilinear", "quadrilinear")
CODE = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
TEXEL_BYTES = {"f32": 16, "f16": 8, "bf16": 8, "e4m3": 4}
# distinct texels read per fragment of a frame of the orbit: what rt_footprint counts there at
# 1920 x 1080 on 1024^2 buckets is 1.35 (quadrilinear); the other filters read fewer
DISTINCT = {"nearest": 0.4, "angular_bilinear": 1.0, "quadrilinear": 1.35}


def listed():
    return [
        # One optimisation step of a small asset through torch.autograd (flat fragments, an atlas
        # tensor as the leaf): the smallest call, where launches and latency count.
        {"name": "quad_autograd_f32", "kind": "autograd", "size": 256, "w": 64, "h": 64, "n": 8, "layout": "atlas",
         "filter": "quadrilinear"},
        # Rendering a camera path: the forward pass of the sphere and plane at 1080p, FP16.
        {"name": "orbit_forward_f16", "kind": "forward", "views": 20, "width": 1920, "height": 1080, "w": 1024,
         "h": 1024, "n": 16, "storage": "f16", "filter": "quadrilinear", "palette": 0, "flat": False},
        # The headline training step: clear, forward, L2 loss and backward over 60 poses.
        {"name": "orbit_step_f16", "kind": "step", "views": 60, "width": 1920, "height": 1080, "w": 1024, "h": 1024,
         "n": 16, "storage": "f16", "filter": "quadrilinear"},
        # Inverse rendering with a loss of the caller's own: the backward alone, ragged frames and
        # odd bucket matrices, BF16.
        {"name": "orbit_backward_bf16", "kind": "backward", "views": 9, "width": 1366, "height": 767, "w": 777,
         "h": 555, "n": 12, "storage": "bf16", "filter": "quadrilinear"},
        # A scene of many assets: 64 textures of uneven resolutions on 4K frames, one launch.
        {"name": "many_objects_4k_f16", "kind": "many", "objects": 64, "views": 2, "width": 3840, "height": 2160,
         "buckets": 384, "storage": "f16", "filter": "quadrilinear"},
        # Serving compressed assets: palette (bucket) compression with E4M3 palettes.
        {"name": "palette_forward_e4m3", "kind": "forward", "views": 20, "width": 1920, "height": 1080, "w": 1024,
         "h": 1024, "n": 16, "storage": "e4m3", "filter": "quadrilinear", "palette": 1024, "flat": False},
        # Normal-mapped surfaces: the world-space lookup, forward and coordinate gradients.
        {"name": "world_step_f16", "kind": "world", "views": 12, "width": 1920, "height": 1080, "w": 1024, "h": 1024,
         "n": 16, "storage": "f16", "filter": "quadrilinear"},
        # Area shadows: several light directions per fragment over 1-bit textures.
        {"name": "area_shadow_bit1", "kind": "shadow", "views": 10, "width": 1920, "height": 1080, "w": 1024,
         "h": 1024, "n": 16, "samples": 4, "filter": "quadrilinear"},
        # Fitting a texture to renders: one Adam step over 32 views, and the reproducible mode's.
        {"name": "fit_step_f32", "kind": "fit", "views": 32, "size": 1024, "w": 512, "h": 512, "n": 16,
         "deterministic": False},
        {"name": "fit_step_deterministic", "kind": "fit", "views": 12, "size": 768, "w": 384, "h": 384, "n": 16,
         "deterministic": True},
        # The asset pipeline: bake a texture from the scene and read its codes back for export,
        {"name": "bake_export_f16", "kind": "bake", "surface": "sphere", "w": 1024, "h": 1024, "n": 16,
         "storage": "f16"},
        # and compress one to a palette (k-means over its buckets).
        {"name": "palette_encode_f16", "kind": "encode", "w": 512, "h": 512, "n": 16, "K": 1024, "iterations": 2,
         "storage": "f16"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _texture_size(rng, lo, hi, most):
    """w, h and n of a texture of at most `most` texels."""
    while True:
        w, h, n = _log(rng, lo, hi), _log(rng, lo, hi), rng.choice((4, 5, 6, 8, 9, 12, 16, 20, 24))
        if w * h * n * n <= most:
            return {"w": w, "h": h, "n": n}


def _frames(rng, views, most):
    """views x height x width of at most `most` fragments; sides of any remainder."""
    while True:
        W = _log(rng, 320, 2560)
        c = {"views": _log(rng, 1, views), "width": W, "height": max(8, int(W * rng.uniform(0.4, 0.9)))}
        if c["views"] * c["width"] * c["height"] <= most:
            return c


def draw(rng):
    kind = rng.choice(("autograd", "forward", "forward", "step", "backward", "many", "world", "shadow", "fit", "fit",
                       "bake", "encode"))
    c = {"kind": kind}
    if kind == "autograd":
        c |= {"size": _log(rng, 48, 1024), **_texture_size(rng, 16, 512, 1 << 25),
              "layout": rng.choice(("atlas", "planes", "quads")), "filter": rng.choice(FILTERS[1:])}
    elif kind in ("forward", "step", "backward", "world"):
        c |= _frames(rng, 20 if kind in ("forward", "step") else 10, 40_000_000)
        c |= _texture_size(rng, 64, 1024, 1 << 28)
        c |= {"storage": rng.choice(STORAGES), "filter": rng.choice(FILTERS + FILTERS[2:] * 2)}
        if kind == "forward":
            c |= {"palette": rng.choice((0, 0, _log(rng, 64, 4096))), "flat": rng.random() < 0.3}
    elif kind == "many":
        c |= _frames(rng, 3, 17_000_000)
        c |= {"objects": _log(rng, 4, 64), "buckets": _log(rng, 128, 384), "storage": rng.choice(STORAGES),
              "filter": rng.choice(FILTERS + FILTERS[2:])}
    elif kind == "shadow":
        c |= _frames(rng, 8, 12_000_000)
        c |= _texture_size(rng, 64, 1024, 1 << 28)
        c |= {"samples": rng.choice((1, 2, 3, 4, 5, 8, 16)), "filter": rng.choice(FILTERS[1:])}
    elif kind == "fit":
        c |= {"views": _log(rng, 2, 24), "size": _log(rng, 128, 1024), **_texture_size(rng, 64, 512, 1 << 26),
              "deterministic": rng.random() < 0.5}
        c["views"] = max(1, min(c["views"], 16_000_000 // c["size"] ** 2))
    elif kind == "bake":
        c |= {"surface": rng.choice(("sphere", "plane")), **_texture_size(rng, 64, 1024, 1 << 28),
              "storage": rng.choice(STORAGES[:3])}
    else:
        c |= _texture_size(rng, 64, 512, 1 << 26)
        c |= {"K": _log(rng, 16, 1024), "iterations": rng.randint(1, 3), "storage": rng.choice(STORAGES[:3])}
    return c


# --------------------------------------------------------------------------- seeded inputs

def _gen(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + salt) % (1 << 62))
    return g


def _smooth(gen, w, h, cells=8):
    grid = torch.rand((1, 1, cells + 1, cells + 1), generator=gen, device=DEV)
    x = torch.nn.functional.interpolate(grid, size=(h, w), mode="bilinear", align_corners=True)[0, 0]
    return (x + 0.05 * (2.0 * torch.rand((h, w), generator=gen, device=DEV) - 1.0)).clamp(0.0, 1.0)


def _centre_directions(n):
    """Direction of every in-bucket texel's centre, (t, s, 3): the inverse of the disc-to-square
    mapping, then of the equisolid projection."""
    b = (2.0 * np.arange(n) + 1.0) / n - 1.0
    bx, by = np.meshgrid(b, b)
    r = np.hypot(bx, by)
    k = np.where(r > 0, np.maximum(np.abs(bx), np.abs(by)) / np.where(r > 0, r, 1.0), 0.0)
    ax, ay = bx * k, by * k
    q = np.sqrt(np.maximum(2.0 - ax * ax - ay * ay, 0.0))
    return np.stack([ax * q, ay * q, 1.0 - ax * ax - ay * ay], axis=-1)


def _lobes(seed, salt, w, h, n):
    """Texels of a texture with one cosine-power lobe per bucket: FP32 planes (n, n, h, w, 4)."""
    gen = _gen(seed, salt)
    rho = torch.rand((h, w, 3), generator=gen, device=DEV)
    z, phi, e = _smooth(gen, w, h), 2.0 * math.pi * _smooth(gen, w, h), _smooth(gen, w, h)
    r = torch.sqrt((1.0 - z * z).clamp_min(0.0))
    d = torch.stack([r * torch.cos(phi), r * torch.sin(phi), z], dim=0)
    p = torch.exp(math.log(200.0) * e)
    I = torch.tensor(_centre_directions(n), dtype=torch.float32, device=DEV)
    T = torch.empty((n, n, h, w, 4), dtype=torch.float32, device=DEV)
    for t in range(n):
        c = (I[t, :, 0, None, None] * d[0] + I[t, :, 1, None, None] * d[1] + I[t, :, 2, None, None] * d[2])
        lobe = torch.pow(c.clamp_min(0.0), p)
        T[t, ..., 3] = lobe
        torch.mul(rho, lobe[..., None], out=T[t, ..., :3])
    return T


def _rays(eye, target, W, H, fov, up):
    eye, target, up = (np.asarray(v, np.float64) for v in (eye, target, up))
    f = (target - eye) / np.linalg.norm(target - eye)
    if abs(float(f @ up)) > 0.999:
        up = np.array([0.0, 1.0, 0.0]) if abs(up[1]) < 0.5 else np.array([1.0, 0.0, 0.0])
    r = np.cross(f, up)
    r /= np.linalg.norm(r)
    u = np.cross(r, f)
    th = math.tan(math.radians(fov) / 2.0)
    x = (2.0 * (torch.arange(W, device=DEV, dtype=torch.float64) + 0.5) / W - 1.0) * (th * W / H)
    y = (1.0 - 2.0 * (torch.arange(H, device=DEV, dtype=torch.float64) + 0.5) / H) * th
    R = [f[k] + x[None, :] * r[k] + y[:, None] * u[k] for k in range(3)]
    inv = torch.rsqrt(R[0] * R[0] + R[1] * R[1] + R[2] * R[2])
    return [c * inv for c in R]


def _orbit(seed, views, W, H, half=4.0):
    """The unit sphere (id 0) on the plane y = -1 (id 1) from an orbit 6 degrees apart."""
    rng = random.Random(seed)
    az0 = rng.uniform(0.0, 2.0 * math.pi)
    uv = torch.empty((views, H, W, 2), device=DEV)
    dr = torch.empty((views, H, W, 3), device=DEV)
    ob = torch.empty((views, H, W), dtype=torch.int32, device=DEV)
    for k in range(views):
        el, az = math.radians(rng.uniform(10.0, 40.0)), az0 + math.radians(6.0) * k
        E = [3.5 * math.cos(el) * math.cos(az), 3.5 * math.sin(el), 3.5 * math.cos(el) * math.sin(az)]
        R = _rays(E, (0.0, 0.0, 0.0), W, H, 60.0, (0.0, 1.0, 0.0))
        b = R[0] * E[0] + R[1] * E[1] + R[2] * E[2]
        disc = b * b - (3.5 ** 2 - 1.0)
        ts = -b - torch.sqrt(disc.clamp_min(0.0))
        sph = (disc >= 0.0) & (ts > 0.0)
        tp = (-1.0 - E[1]) / R[1]
        X, Z = E[0] + tp * R[0], E[2] + tp * R[2]
        pln = (R[1] < 0.0) & (X.abs() <= half) & (Z.abs() <= half) & ~sph
        P = [E[c] + ts * R[c] for c in range(3)]
        inv = torch.rsqrt((P[0] ** 2 + P[1] ** 2 + P[2] ** 2).clamp_min(1e-30))
        P = [c * inv for c in P]
        theta, phi = torch.acos(P[1].clamp(-1.0, 1.0)), torch.atan2(P[2], P[0])
        sp, cp, st, ct = torch.sin(phi), torch.cos(phi), torch.sin(theta), torch.cos(theta)
        V = [E[c] - P[c] for c in range(3)]
        inv = torch.rsqrt(V[0] ** 2 + V[1] ** 2 + V[2] ** 2)
        V = [c * inv for c in V]
        zero = torch.zeros_like(b)

        def pick(s, p):
            return torch.where(sph, s, torch.where(pln, p, zero))

        uv[k, ..., 0] = pick((phi + math.pi) / (2.0 * math.pi), (X + half) / (2.0 * half))
        uv[k, ..., 1] = pick(theta / math.pi, (Z + half) / (2.0 * half))
        dr[k, ..., 0] = pick(-sp * V[0] + cp * V[2], -R[0])
        dr[k, ..., 1] = pick(ct * cp * V[0] - st * V[1] + ct * sp * V[2], -R[2])
        dr[k, ..., 2] = pick(P[0] * V[0] + P[1] * V[1] + P[2] * V[2], -R[1])
        ob[k] = torch.where(sph, 0, torch.where(pln, 1, -1)).to(torch.int32)
    return uv, dr, ob


def _quad(seed, views, size):
    """Views of the square [-1, 1]^2 at z = 0 (id 0) from seeded eyes on the upper hemisphere."""
    rng = random.Random(seed)
    uv = torch.empty((views, size, size, 2), device=DEV)
    dr = torch.empty((views, size, size, 3), device=DEV)
    ob = torch.empty((views, size, size), dtype=torch.int32, device=DEV)
    for k in range(views):
        at = [rng.uniform(-0.5, 0.5), rng.uniform(-0.5, 0.5), 0.0]
        z, phi, dist = rng.uniform(0.2, 1.0), rng.uniform(0.0, 2.0 * math.pi), rng.uniform(2.0, 3.0)
        s = math.sqrt(1.0 - z * z)
        E = [at[0] + dist * s * math.cos(phi), at[1] + dist * s * math.sin(phi), dist * z]
        R = _rays(E, at, size, size, 50.0, (0.0, 0.0, 1.0))
        t = -E[2] / R[2]
        X, Y = E[0] + t * R[0], E[1] + t * R[1]
        hit = (R[2] < 0.0) & (X.abs() <= 1.0) & (Y.abs() <= 1.0)
        zero = torch.zeros_like(t)
        uv[k, ..., 0] = torch.where(hit, (X + 1.0) / 2.0, zero)
        uv[k, ..., 1] = torch.where(hit, (Y + 1.0) / 2.0, zero)
        for c in range(3):
            dr[k, ..., c] = torch.where(hit, -R[c], zero)
        ob[k] = torch.where(hit, 0, -1).to(torch.int32)
    return uv, dr, ob


def _many(seed, objects, views, W, H):
    """Tilted planes in the Voronoi regions of `objects` seeded sites of the screen."""
    rng = np.random.default_rng(seed)
    uv = torch.empty((views, H, W, 2), device=DEV)
    dr = torch.empty((views, H, W, 3), device=DEV)
    ob = torch.empty((views, H, W), dtype=torch.int32, device=DEV)
    th, aspect = math.tan(math.radians(30.0)), W / H
    px = (torch.arange(W, device=DEV, dtype=torch.float64) + 0.5) / W
    py = (torch.arange(H, device=DEV, dtype=torch.float64) + 0.5) / H
    unit = lambda v: v / np.linalg.norm(v)  # noqa: E731
    for k in range(views):
        site = rng.uniform(0.0, 1.0, (objects, 2))
        rows = []  # centre, normal, tangents of each object's plane
        for o in range(objects):
            back = -unit(np.array([(2 * site[o, 0] - 1) * th * aspect, (1 - 2 * site[o, 1]) * th, -1.0]))
            help_ = np.array([0.0, 1.0, 0.0]) if abs(back[1]) < 0.9 else np.array([1.0, 0.0, 0.0])
            e1 = unit(np.cross(help_, back))
            tilt, spin, roll = math.radians(rng.uniform(0, 60)), rng.uniform(0, 2 * math.pi), rng.uniform(0, 2 * math.pi)
            N = math.cos(tilt) * back + math.sin(tilt) * (math.cos(spin) * e1 + math.sin(spin) * np.cross(back, e1))
            t1 = unit(np.cross(N, help_ if abs(N @ help_) < 0.9 else np.array([1.0, 0.0, 0.0])))
            Tx = math.cos(roll) * t1 + math.sin(roll) * np.cross(N, t1)
            rows.append(np.concatenate([-rng.uniform(2.0, 6.0) * back, N, Tx, np.cross(N, Tx)]))
        table = torch.tensor(np.stack(rows), device=DEV)
        sites = torch.tensor(site, device=DEV)
        rays = _rays((0, 0, 0), (0, 0, -1), W, H, 60.0, (0, 1, 0))
        for y0 in range(0, H, 256):
            y1 = min(H, y0 + 256)
            d2 = (px[None, :, None] - sites[:, 0]) ** 2 + (py[y0:y1, None, None] - sites[:, 1]) ** 2
            region = d2.argmin(dim=-1)
            q = table[region]
            C, N, Tx, Ty = (q[..., 3 * m:3 * m + 3] for m in range(4))
            R = torch.stack([c[y0:y1] for c in rays], dim=-1)
            den = (R * N).sum(-1)
            t = (C * N).sum(-1) / den
            rel = t[..., None] * R - C
            front = (t > 0) & (den < 0)
            zero = torch.zeros_like(t)
            for c, T in enumerate((Tx, Ty)):
                uv[k, y0:y1, :, c] = torch.where(front, (0.5 + 0.5 * (rel * T).sum(-1)).clamp(0.0, 1.0), zero)
            for c, T in enumerate((Tx, Ty, N)):
                dr[k, y0:y1, :, c] = torch.where(front, -(R * T).sum(-1), zero)
            ob[k, y0:y1] = torch.where(front, region, torch.full_like(region, -1)).to(torch.int32)
    return uv, dr, ob


def _object_sizes(case, seed):
    rng = np.random.default_rng(seed + 17)
    hi = case["buckets"]
    side = lambda: int(round(math.exp(rng.uniform(math.log(hi / 8), math.log(hi)))))  # noqa: E731
    return [(side(), side(), int(rng.choice((8, 12, 16, 24)))) for _ in range(case["objects"])]


def _palette_index(seed, salt, w, h, K):
    """A bucket map as compression leaves it: smooth regions with per-bucket jitter."""
    gen = _gen(seed, salt)
    x = (K * _smooth(gen, w, h)).to(torch.int32) + torch.randint(0, max(2, K // 16), (h, w), generator=gen, device=DEV,
                                                                 dtype=torch.int32)
    return (x % K).contiguous()


def _normal_map(uv):
    a = 2.0 * math.pi * 8.0 * uv
    N = torch.stack([0.3 * torch.sin(a[..., 0]), 0.3 * torch.cos(a[..., 1]), torch.ones_like(uv[..., 0])], dim=-1)
    return (N / N.norm(dim=-1, keepdim=True)).contiguous()


def _light_directions(seed, dr, samples):
    off = 0.1 * torch.randn((1, samples, 3), generator=_gen(seed, 5), device=DEV)
    L = dr.reshape(-1, 1, 3) + off
    L[..., 2] = L[..., 2].abs()
    return (L / L.norm(dim=2, keepdim=True)).contiguous()


def _target(seed, shape):
    return torch.rand((*shape, 4), generator=_gen(seed, 9), device=DEV)


def _loss_gradient(seed, shape):
    return torch.randn((*shape, 4), generator=_gen(seed, 11), device=DEV)


def _fit_target(seed, uv, dr, ob):
    """Renders of a hidden field: cosine-power lobes modulated over the surface."""
    rng = random.Random(seed + 777)
    out = torch.zeros((*ob.shape, 4), device=DEV)
    for _ in range(4):
        z, phi, p = rng.uniform(0, 1), rng.uniform(0, 2 * math.pi), math.exp(rng.uniform(0, math.log(200.0)))
        r = math.sqrt(1 - z * z)
        c = (r * math.cos(phi)) * dr[..., 0] + (r * math.sin(phi)) * dr[..., 1] + z * dr[..., 2]
        wave = 0.5 + 0.5 * torch.cos(2 * math.pi * (rng.randint(1, 4) * uv[..., 0] + rng.randint(1, 4) * uv[..., 1])
                                     + rng.uniform(0, 2 * math.pi))
        lobe = wave * torch.pow(c.clamp_min(0.0), p)
        out += lobe[..., None] * torch.tensor([rng.uniform(0, 0.25) for _ in range(4)], device=DEV)
    return (out * (ob >= 0)[..., None]).contiguous()


def _fit_start(case, seed):
    return 0.5 * _lobes(seed, 0, case["w"], case["h"], case["n"])


def _bake_scene(seed):
    rng = np.random.default_rng(seed)
    sun = np.array([rng.uniform(-0.6, 0.6), 1.0, rng.uniform(-0.6, 0.6)])
    sun /= np.linalg.norm(sun)
    return {"sphere_centre": [0.0, 0.0, 0.0], "sphere_radius": 1.0, "plane_height": -1.0, "plane_half_extent": 4.0,
            "sphere_albedo": rng.uniform(0.2, 0.9, 3).tolist(), "sphere_reflectance": float(rng.uniform(0.2, 0.6)),
            "plane_albedo": rng.uniform(0.2, 0.9, 3).tolist(), "plane_reflectance": float(rng.uniform(0.2, 0.6)),
            "plane_frequency": float(rng.uniform(2.0, 6.0)), "sun_direction": sun.tolist(),
            "sun_rgb": rng.uniform(0.3, 0.8, 3).tolist(), "sun_exponent": float(rng.integers(4, 17)),
            "sky_zenith": rng.uniform(0.3, 0.8, 3).tolist(), "sky_horizon": rng.uniform(0.3, 0.8, 3).tolist(),
            "ambient": float(rng.uniform(0.1, 0.3)), "fog": float(rng.uniform(0.05, 0.15)), "ray_offset": 1e-4}


LAYOUT = {"atlas": api.RT_LAYOUT_ATLAS, "planes": api.RT_LAYOUT_PLANES, "quads": api.RT_LAYOUT_QUADS}


def _quad_slot(w, i, j):
    return ((j // 2) * ((w + 1) // 2) + i // 2) * 4 + 2 * (j % 2) + i % 2


def _in_layout(planes, layout, w, h, n):
    """A planes tensor in another layout (quads: odd sides padded with zeros)."""
    if layout == "planes":
        return planes
    if layout == "atlas":
        return planes.permute(2, 0, 3, 1, 4).reshape(h * n, w * n, 4).contiguous()
    p = torch.zeros((n, n, h + h % 2, w + w % 2, 4), dtype=planes.dtype, device=DEV)
    p[:, :, :h, :w] = planes
    return p.view(n, n, p.shape[2] // 2, 2, p.shape[3] // 2, 2, 4).transpose(3, 4).contiguous()


def _scene_textures(case, seed, ctx):
    """The two objects' textures of an orbit scene."""
    fmt, w, h, n = api.FORMAT_NAMES[case["storage"]], case["w"], case["h"], case["n"]
    ids = []
    for o in range(2):
        K = case.get("palette", 0)
        if K:
            ids.append(api.rt_create_palette_texture(ctx, w, h, n, K, fmt, api.RT_LAYOUT_PLANES,
                                                     _lobes(seed, o, K, 1, n).view(n, n, K, 4),
                                                     _palette_index(seed, 50 + o, w, h, K)))
        else:
            ids.append(api.rt_create_texture(ctx, w, h, n, fmt, api.RT_LAYOUT_PLANES, _lobes(seed, o, w, h, n)))
    assert ids == [0, 1]
    return ids


def _gradient_buffers(case, ctx):
    return {o: torch.empty(api.layout_shape(api.rt_texture_info(ctx, o)["layout"], case["w"], case["h"], case["n"]),
                           device=DEV) for o in (0, 1)}


def prepare(case, seed):
    kind = case["kind"]
    ctx = api.Context(0)
    S = {"case": case, "ctx": ctx}
    if "filter" in case:
        S["filter"] = api.FILTER_NAMES[case["filter"]]
    if kind == "autograd":
        w, h, n = case["w"], case["h"], case["n"]
        uv, dr, ob = _quad(seed, 1, case["size"])
        S["uv"] = uv.view(-1, 2).requires_grad_()
        S["dir"] = dr.view(-1, 3).requires_grad_()
        S["obj"] = ob.view(-1)
        S["tex"] = _in_layout(_lobes(seed, 0, w, h, n), case["layout"], w, h, n).requires_grad_()
        S["oid"] = api.rt_create_texture(ctx, w, h, n, api.RT_F32, LAYOUT[case["layout"]], S["tex"].detach(),
                                         api.RT_BORROW)
        S["grad_out"] = _loss_gradient(seed, (case["size"] ** 2,))
        return S
    if kind in ("forward", "step", "backward", "world", "shadow"):
        shape = (case["views"], case["height"], case["width"])
        S["uv"], S["dir"], S["obj"] = _orbit(seed, *[shape[k] for k in (0, 2, 1)])
        if kind == "shadow":
            for o in range(2):
                src = _lobes(seed, o, case["w"], case["h"], case["n"])
                src[..., 0] = (src[..., 3] > 0.05).float()
                api.rt_create_texture(ctx, case["w"], case["h"], case["n"], api.RT_BIT1, api.RT_LAYOUT_PLANES, src)
                del src
            S["uv"], S["obj"] = S["uv"].view(-1, 2), S["obj"].view(-1)
            S["dirs"] = _light_directions(seed, S.pop("dir"), case["samples"])
            S["out"] = torch.empty((S["obj"].numel(), 4), device=DEV)
            return S
        _scene_textures(case, seed, ctx)
        if kind == "forward" and case["flat"]:
            S["uv"], S["dir"], S["obj"] = S["uv"].view(-1, 2), S["dir"].view(-1, 3), S["obj"].view(-1)
        if kind != "backward":
            S["out"] = torch.empty((*S["obj"].shape, 4), device=DEV)
        if kind in ("step", "backward", "world"):
            S["duv"], S["ddir"] = torch.empty_like(S["uv"]), torch.empty_like(S["dir"])
        if kind in ("step", "backward"):
            S["dtex"] = _gradient_buffers(case, ctx)
        if kind == "step":
            S["target"], S["sums"] = _target(seed, shape), torch.zeros(2, dtype=torch.float64, device=DEV)
        if kind in ("backward", "world"):
            S["grad_out"] = _loss_gradient(seed, shape)
        if kind == "world":
            S["nrm"] = _normal_map(S["uv"])
            S["dnrm"] = torch.empty_like(S["nrm"])
        return S
    if kind == "many":
        S["uv"], S["dir"], S["obj"] = _many(seed, case["objects"], case["views"], case["width"], case["height"])
        for o, (w, h, n) in enumerate(_object_sizes(case, seed)):
            api.rt_create_texture(ctx, w, h, n, api.FORMAT_NAMES[case["storage"]], api.RT_LAYOUT_PLANES,
                                  _lobes(seed, o, w, h, n))
        S["out"] = torch.empty((*S["obj"].shape, 4), device=DEV)
        return S
    if kind == "fit":
        S["uv"], S["dir"], S["obj"] = _quad(seed, case["views"], case["size"])
        S["target"] = _fit_target(seed, S["uv"], S["dir"], S["obj"])
        S["fit"] = fit.TextureFit(ctx, case["w"], case["h"], case["n"], deterministic=case["deterministic"])
        # a texture some steps into its fit: half the way to another field
        S["fit"].tex.copy_(_in_layout(_fit_start(case, seed), "quads", case["w"], case["h"], case["n"]))
        S["count"] = S["fit"].shaded_count(S["obj"])
        S["out"] = torch.empty((*S["obj"].shape, 4), device=DEV)
        return S
    if kind == "bake":
        S["scene"] = _bake_scene(seed)
        S["surface"] = api.RT_SURFACE_SPHERE if case["surface"] == "sphere" else api.RT_SURFACE_PLANE
        S["oid"] = api.rt_create_texture(ctx, case["w"], case["h"], case["n"], api.FORMAT_NAMES[case["storage"]])
        return S
    S["oid"] = api.rt_create_texture(ctx, case["w"], case["h"], case["n"], api.FORMAT_NAMES[case["storage"]],
                                     api.RT_LAYOUT_PLANES, _lobes(seed, 0, case["w"], case["h"], case["n"]))
    S["seed"] = int(seed)
    return S


def run(S):
    kind, ctx = S["case"]["kind"], S["ctx"]
    if kind == "autograd":
        out = autograd.shade(ctx, S["uv"], S["dir"], S["obj"], S["filter"], {S["oid"]: S["tex"]})
        return (out.detach(), *torch.autograd.grad(out, (S["tex"], S["uv"], S["dir"]), S["grad_out"]))
    if kind == "forward":
        call = api.rt_shade if S["case"]["flat"] else api.rt_shade_batched
        return call(ctx, S["uv"], S["dir"], S["obj"], S["filter"], S["out"])
    if kind == "many":
        return api.rt_shade_batched(ctx, S["uv"], S["dir"], S["obj"], S["filter"], S["out"])
    if kind == "step":
        S["sums"].zero_()
        api.rt_zero_texture_grads(ctx, S["dtex"])
        api.rt_shade_batched_l2_step(ctx, S["uv"], S["dir"], S["obj"], S["filter"], S["target"], 1.0, S["out"],
                                     S["sums"], S["dtex"], S["duv"], S["ddir"], api.RT_ACCUMULATE_TEXELS)
        return S["out"], S["sums"], S["dtex"][0], S["dtex"][1], S["duv"], S["ddir"]
    if kind == "backward":
        api.rt_shade_batched_backward(ctx, S["uv"], S["dir"], S["obj"], S["filter"], S["grad_out"], S["dtex"],
                                      S["duv"], S["ddir"])
        return S["dtex"][0], S["dtex"][1], S["duv"], S["ddir"]
    if kind == "world":
        api.rt_shade_world_batched(ctx, S["uv"], S["dir"], S["nrm"], S["obj"], S["filter"], S["out"])
        api.rt_shade_world_batched_backward(ctx, S["uv"], S["dir"], S["nrm"], S["obj"], S["filter"], S["grad_out"],
                                            None, S["duv"], S["ddir"], S["dnrm"])
        return S["out"], S["duv"], S["ddir"], S["dnrm"]
    if kind == "shadow":
        return api.rt_shade_multi(ctx, S["uv"], S["dirs"], S["obj"], S["filter"], S["out"])
    if kind == "fit":
        f = S["fit"]
        loss = f.step(S["uv"], S["dir"], S["obj"], S["target"], S["count"], S["out"])
        return loss, S["out"], f.grad, f.m, f.v, f.tex
    if kind == "bake":
        api.rt_bake(ctx, S["oid"], S["surface"], S["scene"])
        codes, _ = api.rt_read_texture(ctx, S["oid"])
        return codes.view(CODE[S["case"]["storage"]])
    C, index, sse = api.palette_encode(ctx, S["oid"], S["case"]["K"], S["case"]["iterations"], seed=S["seed"])
    return C, index, sse


# --------------------------------------------------------------------------- work

def _touched(case, F, texels):
    return min(int(F * DISTINCT[case["filter"]]), texels)


def work(case):
    kind = case["kind"]
    taps = {"nearest": 1, "angular_bilinear": 4, "quadrilinear": 16}[case.get("filter", "quadrilinear")]
    if kind == "autograd":
        F, texels = case["size"] ** 2, case["w"] * case["h"] * case["n"] ** 2
        # forward and backward: G-buffer once, colours out, their gradient in, UV / direction gradients out
        return {"bytes": F * (24 + 16 + 16 + 20) + 16 * _touched(case, F, texels) + 16 * texels,
                "flops": F * (200 + taps * 8 * 3)}
    if kind in ("forward", "step", "backward", "world", "many", "shadow"):
        F = case["views"] * case["width"] * case["height"]
        if kind == "shadow":
            S = case["samples"]
            return {"bytes": F * (8 + 4 + 16 + 12 * S) + 2 * case["w"] * case["h"] * case["n"] ** 2 // 8,
                    "flops": F * S * (60 + taps * 8)}
        tb = TEXEL_BYTES[case["storage"]]
        if kind == "many":
            return {"bytes": F * 40 + tb * _touched(case, F, 1 << 62), "flops": F * (60 + taps * 8)}
        if case.get("palette"):
            K = case["palette"]
            return {"bytes": F * 40 + 2 * (tb * K * case["n"] ** 2 + 4 * K + 4 * case["w"] * case["h"]),
                    "flops": F * (60 + taps * 8)}
        texels = 2 * case["w"] * case["h"] * case["n"] ** 2
        read = tb * _touched(case, F, texels)
        if kind == "forward":
            return {"bytes": F * 40 + read, "flops": F * (60 + taps * 8)}
        if kind == "step":
            return {"bytes": F * (24 + 16 + 16 + 20) + read + 16 * texels, "flops": F * (200 + taps * 24)}
        if kind == "backward":
            return {"bytes": F * (24 + 16 + 20) + read + 16 * texels, "flops": F * (200 + taps * 16)}
        return {"bytes": F * (36 + 16 + 16 + 32) + read, "flops": F * (260 + taps * 16)}
    texels = case["w"] * case["h"] * case["n"] ** 2
    if kind == "fit":
        F = case["views"] * case["size"] ** 2
        # views in, colours out; the texture, its gradient and the two moments read and written
        return {"bytes": F * (24 + 16 + 16) + texels * 16 * 7, "flops": F * (100 + taps * 24) + texels * 4 * 12}
    if kind == "bake":
        return {"bytes": texels * TEXEL_BYTES[case["storage"]], "flops": texels * 128}
    B, D, K, it = case["w"] * case["h"], case["n"] ** 2 * 4, case["K"], case["iterations"]
    return {"bytes": (2 * it + 1) * B * D * (4 if case["storage"] == "f32" else 2) + K * D * 4,
            "flops": 2.0 * B * K * D * (it + 1)}


# --------------------------------------------------------------------------- the same results in 64 bits

class _Stored:
    """The values a texture holds after encoding, gathered as FP64 (n n h w planes order)."""

    def __init__(self, src, storage, w, h, n, index=None):
        self.w, self.h, self.n, self.index = w, h, n, index  # w x h: the bucket matrix
        self.plane = src.shape[2] * src.shape[3]
        self.scale = None
        flat = src.reshape(-1, 4)
        if storage == "e4m3":
            amax = src.abs().amax(dim=(0, 1, 4)).reshape(-1)
            self.scale = torch.where(amax == 0, torch.ones_like(amax), amax / torch.full_like(amax, 448.0))
            q = (src.reshape(n * n, self.plane, 4) / self.scale[None, :, None]).clamp(-448.0, 448.0)
            self.codes = q.to(torch.float8_e4m3fn).view(torch.uint8).reshape(-1, 4)
        elif storage == "bit1":
            self.codes = (flat[:, 0] >= 0.5).to(torch.uint8)
        else:
            self.codes = flat.to(CODE[storage])
        self.storage = storage

    def slot(self, i, j):
        b = j * self.w + i
        return b if self.index is None else self.index.reshape(-1)[b].long()

    def take(self, p, i, j):
        b = self.slot(i, j)
        c = self.codes[p * self.plane + b]
        if self.storage == "e4m3":
            return c.view(torch.float8_e4m3fn).double() * self.scale[b].double()[:, None]
        return c.double()[:, None].expand(-1, 4) if self.storage == "bit1" else c.double()


def _square(h):
    ax, ay = h[:, 0].abs(), h[:, 1].abs()
    m = torch.where(ax >= ay, ax, ay)
    ok = m >= 1e-18
    x, y, z = (torch.where(ok, h[:, k] / torch.where(ok, m, 1.0), 0.0) for k in range(3))
    g2 = torch.where(ok, x * x + y * y, 1.0)
    k = math.sqrt(2.0) * torch.sqrt(g2 / (g2 + z * z))
    return x * k, y * k


def _axis(c, size, linear):
    """The taps of a continuous coordinate: (index, weight) pairs."""
    f = torch.floor(c.detach())
    if not linear:
        return [(f.clamp(0, size - 1).long(), None)]
    w = c - f
    return [(f.clamp(0, size - 1).long(), 1.0 - w), ((f + 1).clamp(0, size - 1).long(), w)]


def _lookup(tex, uv, half, filt, g=None, dtex=None, grad_slot=None):
    """Colours (F, 4) of fragments of one object; with g = dL/dout also the gradients of uv and
    half, the texel gradients added to dtex at grad_slot(plane, i, j)."""
    need = g is not None
    uv = uv.double().detach().requires_grad_(need)
    half = half.double().detach().requires_grad_(need)
    quad, near = filt == "quadrilinear", filt == "nearest"
    w, h, n = tex.w, tex.h, tex.n
    if quad:
        cu, cv = (uv[:, 0] * w - 0.5).clamp(-1.0, w), (uv[:, 1] * h - 0.5).clamp(-1.0, h)
    else:
        cu, cv = (uv[:, 0] * w).clamp(0.0, w), (uv[:, 1] * h).clamp(0.0, h)
    hi = 1.0 - 1.0 / n
    cs, ct = ((b.clamp(-hi, hi) + 1.0) * (n / 2.0) for b in _square(half))
    if not near:
        cs, ct = (cs - 0.5).clamp(0.0, n - 1.0), (ct - 0.5).clamp(0.0, n - 1.0)
    out = torch.zeros((uv.shape[0], 4), dtype=torch.float64, device=DEV)
    total = 0.0
    for j, wv in _axis(cv, h, quad):
        for i, wu in _axis(cu, w, quad):
            for t, wt in _axis(ct, n, not near):
                for s, ws in _axis(cs, n, not near):
                    wgt = torch.ones_like(cu)
                    for x in (wv, wu, wt, ws):
                        wgt = wgt if x is None else wgt * x
                    T = tex.take(t * n + s, i, j)
                    out += wgt.detach()[:, None] * T
                    if need:
                        total = total + (wgt * (T * g).sum(-1)).sum()
                        if dtex is not None:
                            dtex.index_add_(0, grad_slot(t * n + s, i, j), wgt.detach()[:, None] * g)
    if not need:
        return out
    if not near:
        gu, gh = torch.autograd.grad(total, (uv, half), allow_unused=True)
    else:
        gu = gh = None
    zeros = torch.zeros_like
    return out, zeros(uv) if gu is None else gu, zeros(half) if gh is None else gh


def _over(textures, uv, half, ob, filt, grad=None, dtex=None, slots=None, chunk=2_000_000):
    """_lookup over flat fragments of several objects.  grad(out, where) gives dL/dout."""
    F = ob.numel()
    out = torch.zeros((F, 4), dtype=torch.float64, device=DEV)
    gu = torch.zeros((F, 2), dtype=torch.float64, device=DEV) if grad else None
    gh = torch.zeros((F, 3), dtype=torch.float64, device=DEV) if grad else None
    for f0 in range(0, F, chunk):
        part = ob[f0:f0 + chunk]
        for o, tex in enumerate(textures):
            at = f0 + (part == o).nonzero()[:, 0]
            if not at.numel():
                continue
            if not grad:
                out[at] = _lookup(tex, uv[at], half[at], filt)
                continue
            with torch.no_grad():
                g = grad(_lookup(tex, uv[at], half[at], filt), at)
            out[at], gu[at], gh[at] = _lookup(tex, uv[at], half[at], filt, g, dtex[o] if dtex else None,
                                              slots[o] if slots else None)
    return out, gu, gh


def _up(d):
    return d + torch.tensor([0.0, 0.0, 1.0], device=DEV, dtype=torch.float64)


def _quads(w, h, n):
    P = 4 * ((w + 1) // 2) * ((h + 1) // 2)
    return n * n * P, lambda p, i, j: p * P + _quad_slot(w, i, j)


def _exact_bake(case, seed):
    sc, w, h, n = _bake_scene(seed), case["w"], case["h"], case["n"]
    f32 = lambda v: torch.tensor(np.asarray(v, np.float32).astype(np.float64), device=DEV)  # noqa: E731
    S = {k: f32(v) for k, v in sc.items()}
    d64 = {"dtype": torch.float64, "device": DEV}
    u, v = (torch.arange(w, **d64) + 0.5) / w, (torch.arange(h, **d64) + 0.5) / h
    one, zero = torch.ones((h, w), **d64), torch.zeros((h, w), **d64)
    dot = lambda a, b: a[0] * b[0] + a[1] * b[1] + a[2] * b[2]  # noqa: E731

    def lit(N):
        return S["ambient"] + (1 - S["ambient"]) * dot(N, S["sun_direction"]).clamp_min(0.0)

    def plane_albedo(x, z):
        f = S["plane_frequency"]
        m = 0.75 + 0.25 * torch.cos(f * x) * torch.cos(f * z)
        return [m * S["plane_albedo"][c] for c in range(3)]

    if case["surface"] == "sphere":
        sp, cp = torch.sin(2 * math.pi * u - math.pi)[None, :] * one, torch.cos(2 * math.pi * u - math.pi)[None, :] * one
        st, ct = torch.sin(math.pi * v)[:, None] * one, torch.cos(math.pi * v)[:, None] * one
        N, T, B = [st * cp, ct, st * sp], [-sp, zero, cp], [ct * cp, -st, ct * sp]
        P = [S["sphere_centre"][c] + S["sphere_radius"] * N[c] for c in range(3)]
        base, refl = [lit(N) * S["sphere_albedo"][c] for c in range(3)], S["sphere_reflectance"]
    else:
        e = S["plane_half_extent"]
        P = [(2 * e * u - e)[None, :] * one, S["plane_height"] * one, (2 * e * v - e)[:, None] * one]
        T, B, N = [one, zero, zero], [zero, zero, one], [zero, one, zero]
        base, refl = plane_albedo(P[0], P[2]), S["plane_reflectance"]
        base = [lit(N) * b for b in base]
    I = torch.tensor(_centre_directions(n), **d64)
    out = torch.empty((h, n, w, n, 4), dtype=torch.float64, device=DEV)
    o = [P[c] - S["sphere_centre"][c] for c in range(3)]
    q = dot(o, o) - S["sphere_radius"] ** 2
    inf = torch.full_like(one, math.inf)
    for t in range(n):
        for s in range(n):
            R = (-I[t, s, 0], -I[t, s, 1], I[t, s, 2])
            d = [R[0] * T[c] + R[1] * B[c] + R[2] * N[c] for c in range(3)]
            b = dot(o, d)
            disc = b * b - q
            ts = torch.where(disc > 0, -b - torch.sqrt(disc.clamp_min(0.0)), inf)
            ts = torch.where(ts > S["ray_offset"], ts, inf)
            tp = torch.where(d[1] != 0, (S["plane_height"] - P[1]) / torch.where(d[1] != 0, d[1], one), inf)
            tp = torch.where(tp > S["ray_offset"], tp, inf)
            plane = tp < ts
            tb = torch.where(plane, tp, ts)
            hit = torch.isfinite(tb)
            tb = torch.where(hit, tb, zero)
            X = [P[c] + tb * d[c] for c in range(3)]
            Nh = [(X[c] - S["sphere_centre"][c]) / S["sphere_radius"] for c in range(3)]
            ls, lp, ap = lit(Nh), lit([zero, one, zero]), plane_albedo(X[0], X[2])
            sun = torch.pow(dot(d, S["sun_direction"]).clamp_min(0.0), S["sun_exponent"])
            g = torch.where(hit, torch.exp(-S["fog"] * tb), zero)
            for c in range(3):
                sky = (S["sky_horizon"][c] + (S["sky_zenith"][c] - S["sky_horizon"][c]) * (0.5 + 0.5 * d[1])
                       + S["sun_rgb"][c] * sun)
                C = torch.where(plane, lp * ap[c], ls * S["sphere_albedo"][c])
                out[:, t, :, s, c] = base[c] + refl * (g * C + (1 - g) * sky)
            out[:, t, :, s, 3] = g
    return out.view(h * n, w * n, 4)


def _exact_fit(case, seed):
    w, h, n = case["w"], case["h"], case["n"]
    uv, dr, ob = _quad(seed, case["views"], case["size"])
    target, shape = _fit_target(seed, uv, dr, ob).view(-1, 4), ob.shape
    uv, dr, ob = uv.view(-1, 2), dr.view(-1, 3), ob.view(-1)
    count = int((ob >= 0).sum())
    texels, slot = _quads(w, h, n)
    grad = torch.zeros((texels, 4), dtype=torch.float64, device=DEV)
    start = _fit_start(case, seed)
    tex = _Stored(start, "f32", w, h, n)
    scale = 1.0 / (4.0 * max(count, 1))
    out, _, _ = _over([tex], uv, _up(dr.double()), ob, "quadrilinear",
                      lambda c, at: scale * (c - target[at].double()), [grad], [slot])
    loss = 0.5 * scale * ((out - target.double()) ** 2 * (ob >= 0)[:, None]).sum()
    m, v = 0.1 * grad, 0.001 * grad * grad
    p = _in_layout(start, "quads", w, h, n).view(-1, 4).double()
    p -= 1e-2 * (m / 0.1) / (torch.sqrt(v / 0.001) + 1e-8)
    form = api.layout_shape(api.RT_LAYOUT_QUADS, w, h, n)
    return (loss, out.view(*shape, 4), *(x.view(form) for x in (grad, m, v, p)))


def exact(case, seed):
    kind = case["kind"]
    if kind == "encode":  # integer choices decide the rest: nothing here has one value in 64 bits
        return None
    if kind == "bake":
        return _exact_bake(case, seed)
    if kind == "fit":
        return _exact_fit(case, seed)
    filt = case["filter"]
    if kind == "autograd":
        w, h, n = case["w"], case["h"], case["n"]
        uv, dr, ob = _quad(seed, 1, case["size"])
        g = _loss_gradient(seed, (case["size"] ** 2,)).double()
        tex = _Stored(_lobes(seed, 0, w, h, n), "f32", w, h, n)
        dtex = torch.zeros((n * n * w * h, 4), dtype=torch.float64, device=DEV)
        out, gu, gh = _over([tex], uv.view(-1, 2), _up(dr.view(-1, 3).double()), ob.view(-1), filt,
                            lambda c, at: g[at], [dtex], [lambda p, i, j: p * (w * h) + j * w + i])
        return out, _in_layout(dtex.view(n, n, h, w, 4), case["layout"], w, h, n), gu, gh
    if kind == "many":
        uv, dr, ob = _many(seed, case["objects"], case["views"], case["width"], case["height"])
        tex = [_Stored(_lobes(seed, o, w, h, n), case["storage"], w, h, n)
               for o, (w, h, n) in enumerate(_object_sizes(case, seed))]
        out = _over(tex, uv.view(-1, 2), _up(dr.view(-1, 3).double()), ob.view(-1), filt, chunk=8_000_000)[0]
        return out.view(*ob.shape, 4)
    w, h, n = case["w"], case["h"], case["n"]
    uv, dr, ob = _orbit(seed, case["views"], case["width"], case["height"])
    shape = ob.shape
    if kind == "shadow":
        tex = []
        for o in range(2):
            src = _lobes(seed, o, w, h, n)
            src[..., 0] = (src[..., 3] > 0.05).float()
            tex.append(_Stored(src, "bit1", w, h, n))
            del src
        L = _light_directions(seed, dr, case["samples"])
        uv, ob = uv.view(-1, 2), ob.view(-1)
        out = torch.zeros((ob.numel(), 4), dtype=torch.float64, device=DEV)
        for k in range(case["samples"]):
            out += _over(tex, uv, _up(L[:, k].double()), ob, filt)[0]
        return out / case["samples"]
    K = case.get("palette", 0)
    tex = [_Stored(_lobes(seed, o, K, 1, n), case["storage"], w, h, n, _palette_index(seed, 50 + o, w, h, K)) if K
           else _Stored(_lobes(seed, o, w, h, n), case["storage"], w, h, n) for o in range(2)]
    half = _up(dr.view(-1, 3).double()) if kind != "world" else dr.view(-1, 3).double() + _normal_map(uv).view(-1, 3)
    uv, ob = uv.view(-1, 2), ob.view(-1)
    if kind == "forward":
        out = _over(tex, uv, half, ob, filt)[0]
        return out if case["flat"] else out.view(*shape, 4)
    texels, slot = _quads(w, h, n)
    form = api.layout_shape(api.RT_LAYOUT_QUADS, w, h, n)
    dtex = None if kind == "world" else [torch.zeros((texels, 4), dtype=torch.float64, device=DEV) for _ in range(2)]
    if kind == "step":
        target = _target(seed, shape).view(-1, 4)
        grad = lambda c, at: c - target[at].double()  # noqa: E731
    else:
        g = _loss_gradient(seed, shape).view(-1, 4)
        grad = lambda c, at: g[at].double()  # noqa: E731
    out, gu, gh = _over(tex, uv, half, ob, filt, grad, dtex, [slot, slot])
    gu, gh, out = gu.view(*shape, 2), gh.view(*shape, 3), out.view(*shape, 4)
    if kind == "world":
        return out, gu, gh, gh
    if kind == "backward":
        return dtex[0].view(form), dtex[1].view(form), gu, gh
    r = (out.view(-1, 4) - target.double()) * (ob >= 0)[:, None]
    sums = torch.stack([(r * r).sum(), (ob >= 0).sum().double()])
    return out, sums, dtex[0].view(form), dtex[1].view(form), gu, gh
