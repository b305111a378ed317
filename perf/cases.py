"""The work a user has this library do, as cases that can be timed and checked.

A case is one pass through a public entry point on inputs made from a seed:

  view     Renderer.render_view: one view as a replay of the captured graph, or (graphs
           False) the plain render_view call
  serve    ViewServer.run: a burst of views of mixed sizes from one resident scene
  maps     render_gradients: the composite alone (every pixel of the planes)
  project  the projection alone, with all its outputs
  poisson  poisson_reconstruct: gradient maps to image
  rho      poisson_reconstruct_rho: a Laplacian field (with the hard threshold) to image
  train    autograd.render_view, a mean squared error and its backward

`exact` computes the same in 64 bits with plain torch: the projection and the composite
by their definitions tile by tile, the Neumann solve by an FFT of the even extension, the
parameter gradients by torch's autograd.
"""
from __future__ import annotations

import math
import types

import numpy as np
import torch

import paper_2405_05446_gb300 as G
from paper_2405_05446_gb300 import autograd as A
from paper_2405_05446_gb300 import scenes as S
from paper_2405_05446_gb300 import serving as SV

STORAGE = {"f32": 0, "bf16": 1, "f16": 2}
TILE = 16
ALPHA_MIN, ALPHA_MAX, T_MIN, DILATION = 1.0 / 255.0, 0.99, 1e-4, 0.3
PARAMS = ("mean", "scale", "quat", "opacity", "grad")


def listed():
    return [
        # the smallest view anyone renders (the smoke view): launches and latency
        {"name": "view_tiny64", "kind": "view", "n": 1000, "w": 64, "h": 64, "c": 3,
         "scene": "tiny", "attr": "gradient", "graphs": True},
        # the headline view: 200k Gaussians at 1920x1080, replayed
        {"name": "view_1080p", "kind": "view", "n": 200_000, "w": 1920, "h": 1080, "c": 3,
         "scene": "prims", "attr": "gradient", "graphs": True},
        # the largest view: 1M Gaussians at 3840x2160
        {"name": "view_4k", "kind": "view", "n": 1_000_000, "w": 3840, "h": 2160, "c": 3,
         "scene": "prims", "attr": "gradient", "graphs": True},
        # the paper-literal Laplacian attribute through the plain call (no whole-view graph)
        {"name": "view_lap_1080p", "kind": "view", "n": 200_000, "w": 1920, "h": 1080, "c": 3,
         "scene": "prims", "attr": "laplacian", "graphs": False},
        # a server with a resident 400k scene and ten requests over its five image sizes
        {"name": "serve_mix", "kind": "serve", "n": 400_000, "requests": 10, "c": 3,
         "wmax": 3840, "storage": "bf16"},
        # gradient maps for another consumer (four channels, ragged size)
        {"name": "maps_ragged", "kind": "maps", "n": 300_000, "w": 1237, "h": 711, "c": 4,
         "scene": "prims", "attr": "gradient"},
        # projection of a large scene (culling, statistics, densification use its outputs)
        {"name": "project_1m", "kind": "project", "n": 1_000_000, "w": 1920, "h": 1080, "c": 3},
        # one small image from its gradients: an interactive edit
        {"name": "poisson_small", "kind": "poisson", "w": 128, "h": 96, "c": 1,
         "storage": "f32", "mask": False, "nu1": 2, "nu2": 1},
        # a full-size image from sparse maps (tile mask)
        {"name": "poisson_1080p", "kind": "poisson", "w": 1920, "h": 1080, "c": 3,
         "storage": "f32", "mask": True, "nu1": 2, "nu2": 1},
        # an odd-sized photograph, 16-bit storage of the corrections
        {"name": "poisson_odd", "kind": "poisson", "w": 1355, "h": 757, "c": 3,
         "storage": "bf16", "mask": False, "nu1": 2, "nu2": 1},
        # a splatted Laplacian field at 4K with the hard threshold, one channel
        {"name": "rho_4k", "kind": "rho", "w": 3840, "h": 2160, "c": 1, "storage": "f16",
         "threshold": 0.004},
        # one view of the training workload: forward, loss, backward
        {"name": "train_720p", "kind": "train", "n": 500_000, "w": 1280, "h": 720, "c": 3,
         "attr": "gradient"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["view", "view", "view", "serve", "maps", "project", "poisson", "poisson",
                       "rho", "train"])
    w = _log_int(rng, 64, 3840)
    h = max(48, min(2160, int(w * rng.uniform(0.4, 1.2))))
    n = min(_log_int(rng, 1000, 1_000_000), 16 * w * h)
    c = rng.choice([1, 3, 3, 4])
    attr = rng.choice(["gradient", "gradient", "gradient", "laplacian"])
    storage = rng.choice(["f32", "f32", "bf16", "f16"])
    if kind == "serve":
        return {"kind": kind, "n": _log_int(rng, 50_000, 400_000), "requests": rng.randint(4, 10),
                "c": 3, "wmax": rng.choice([512, 1280, 1920, 3840]), "storage": storage}
    if kind == "project":
        return {"kind": kind, "n": _log_int(rng, 1000, 1_000_000), "w": w, "h": h, "c": c}
    if kind == "poisson":
        nu1, nu2 = rng.choice([(2, 1), (2, 1), (2, 1), (2, 1), (2, 2), (1, 1)])
        return {"kind": kind, "w": w, "h": h, "c": c, "storage": storage,
                "mask": rng.random() < 0.5, "nu1": nu1, "nu2": nu2}
    if kind == "rho":
        return {"kind": kind, "w": w, "h": h, "c": c, "storage": storage,
                "threshold": rng.choice([0.0, 0.004])}
    if kind == "train":
        w, h = min(w, 1600), min(h, 900)
        return {"kind": kind, "n": min(n, 500_000), "w": w, "h": h, "c": min(c, 3), "attr": attr}
    out = {"kind": kind, "n": n, "w": w, "h": h, "c": min(c, 3) if kind == "view" else c,
           "scene": "prims", "attr": attr}
    if kind == "view":
        out["graphs"] = rng.random() < 0.6
    return out


# ------------------------------------------------------------------ inputs

def _ppg(w, h):
    """Pair capacity per Gaussian: splats cover more tiles as the image grows."""
    return 32 if w > 2560 or w * h > 4_000_000 else 16


def _scene(case, seed):
    w, h = case.get("w", 1920), case.get("h", 1080)
    cam = S.metric_camera(w, h)
    if case.get("scene") == "tiny":
        sc = S.tiny_scene(seed, n=case["n"], channels=case["c"])
    else:
        sc = S.primitives_scene(seed, n=case["n"], n_prims=50 if case["n"] >= 500_000 else 20,
                                channels=case["c"], orient_camera=cam)
    if case.get("attr") == "laplacian":
        sc = S.with_laplacian_attribute(sc, seed)
    return sc, cam


def _means(c):
    return [0.5, 0.4, 0.6, 0.45][:c]


def _photo(c, h, w, seed, device="cuda"):
    """An image: a smooth part, a few hard edges and some noise, about [0, 1]."""
    gen = torch.Generator(device=device)
    gen.manual_seed(seed)
    y = torch.linspace(0.0, 1.0, h, device=device)[:, None]
    x = torch.linspace(0.0, 1.0, w, device=device)[None, :]
    img = torch.empty((c, h, w), device=device)
    for k in range(c):
        p = torch.rand(8, generator=gen, device=device).tolist()
        a = 0.5 + 0.25 * torch.sin(6.0 * (p[0] + 0.3) * x + 6.0 * p[1]) * torch.cos(5.0 * (p[2] + 0.3) * y)
        a = a + 0.2 * ((x - p[3]) * (p[4] + 0.2) + (y - p[5]) * (p[6] - 0.5) > 0).float()
        a = a - 0.15 * ((x - p[6]) ** 2 + (y - p[7]) ** 2 < 0.04).float()
        img[k] = a
    return img + 0.02 * torch.randn((c, h, w), generator=gen, device=device)


def _gradient_maps(img):
    c, h, w = img.shape
    maps = torch.zeros((c, 2, h, w), device=img.device, dtype=img.dtype)
    maps[:, 0, :, :-1] = img[:, :, 1:] - img[:, :, :-1]
    maps[:, 1, :-1, :] = img[:, 1:, :] - img[:, :-1, :]
    return maps


def _poisson_inputs(case, seed):
    c, h, w = case["c"], case["h"], case["w"]
    maps = _gradient_maps(_photo(c, h, w, seed)).contiguous()
    mask = None
    if case["mask"]:  # three tiles in four hold a splat
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed + 1)
        t = ((h + TILE - 1) // TILE, (w + TILE - 1) // TILE)
        mask = (torch.rand(t, generator=gen, device="cuda") < 0.75).to(torch.uint8)
    return maps, mask


def _rho_input(case, seed):
    """A Laplacian field as splats give it: sparse blobs a few pixels wide with Laplace
    amplitudes, whose sum is not zero."""
    c, h, w = case["c"], case["h"], case["w"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    u = torch.rand((c, h, w), generator=gen, device="cuda") * 2.0 - 1.0
    amp = -0.05 * torch.sign(u) * torch.log1p(-u.abs().clamp_max(1.0 - 1e-6))
    rho = amp * (torch.rand((c, h, w), generator=gen, device="cuda") < 0.01)
    tap = torch.exp(-(torch.arange(-8, 9, device="cuda") ** 2) / 18.0).tolist()
    for dim, size in ((1, h), (2, w)):
        pad = torch.nn.functional.pad(rho, (8, 8, 0, 0) if dim == 2 else (0, 0, 8, 8))
        rho = sum(t * pad.narrow(dim, k, size) for k, t in enumerate(tap))
    return rho.contiguous()


def _requests(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    sizes = [s for s in SV.SIZES if s[0] <= case["wmax"]]
    return [SV.Request(0, S.sphere_camera(rng, *sizes[i % len(sizes)]), 0.0, keep=True)
            for i in range(case["requests"])]


def _sopts(case):
    kw = {"storage": STORAGE[case.get("storage", "f32")]}
    for k in ("nu1", "nu2"):
        if k in case:
            kw[k] = case[k]
    if case.get("threshold"):
        kw["rho_threshold"] = case["threshold"]
    return G.solver_opts(**kw)


def prepare(case, seed):
    kind, c = case["kind"], case["c"]
    st = types.SimpleNamespace(kind=kind, mean=_means(c))
    if kind == "serve":
        sc, _ = _scene(case, seed)
        st.reqs = _requests(case, seed)
        st.server = SV.ViewServer(budget_bytes=60 << 30, slots=4, sopts=_sopts(case))
        st.server.add_scene(0, sc, st.mean)
        st.server.warm(st.reqs)
        return st
    w, h = case["w"], case["h"]
    st.sopts = _sopts(case)
    if kind in ("poisson", "rho"):
        st.mask = None
        if kind == "poisson":
            st.field, st.mask = _poisson_inputs(case, seed)
        else:
            st.field = _rho_input(case, seed)
        st.ws = torch.empty(G.workspace_size(0, c, w, h, None, st.sopts), dtype=torch.uint8, device="cuda")
        st.out = torch.empty((c, h, w), device="cuda")
        return st
    sc, st.cam = _scene(case, seed)
    st.ropts = G.raster_opts(pairs_per_gaussian=_ppg(w, h))
    st.g = G.gaussians_to_device(sc)
    if kind == "train":
        st.params = [getattr(st.g, k).requires_grad_(True) for k in PARAMS]
        st.target = _photo(c, h, w, seed + 2)
        return st
    if kind == "view":
        st.renderer = G.Renderer(sc.n, c, w, h, st.ropts, st.sopts, graphs=case["graphs"])
        st.out = torch.empty((c, h, w), device="cuda")
        return st
    st.ws = torch.empty(G.workspace_size(sc.n, c, w, h, st.ropts, None), dtype=torch.uint8, device="cuda")
    if kind == "maps":
        shape = (c, h, w) if case["attr"] == "laplacian" else (c, 2, h, w)
        st.out = torch.empty(shape, device="cuda")
    else:
        st.out = {"mean2d": torch.empty((sc.n, 2), device="cuda"),
                  "cov2d": torch.empty((sc.n, 3), device="cuda"),
                  "depth": torch.empty(sc.n, device="cuda"),
                  "rect": torch.empty((sc.n, 4), dtype=torch.int32, device="cuda")}
    return st


def run(st):
    if st.kind == "view":
        return st.renderer.render_view(st.g, st.cam, st.mean, st.out)
    if st.kind == "serve":
        return [r.image for r in st.server.run(st.reqs, realtime=False)]
    if st.kind == "maps":
        G.render_gradients(st.g, st.cam, st.out, st.ws, ropts=st.ropts)
        return st.out
    if st.kind == "project":
        G.project(st.g, st.cam, st.ws, st.ropts, **st.out)
        return st.out
    if st.kind == "poisson":
        G.poisson_reconstruct(st.field, st.mean, st.out, st.ws, st.mask, st.sopts)
        return st.out
    if st.kind == "rho":
        G.poisson_reconstruct_rho(st.field, st.mean, st.out, st.ws, sopts=st.sopts)
        return st.out
    for p in st.params:
        p.grad = None
    img = A.render_view(*st.params, st.cam, st.mean, st.ropts, st.sopts)
    loss = ((img - st.target) ** 2).mean()
    loss.backward()
    out = {"d_" + k: p.grad for k, p in zip(PARAMS, st.params)}
    out["image"] = img.detach()
    return out


# ------------------------------------------------------------------ what a pass cannot do without

def _gaussian_bytes(n, q):
    return 4.0 * n * (11 + q)


def _composite_flops(n, w, q):
    # projected sigma 0.0024 w px; a splat reaches alpha_min over about 20 sigma^2 (+ the
    # dilation's share) pixels; an exponent, an exponential and q multiply-adds each
    px = 20.0 * (0.0024 * w) ** 2 + 15.0 * DILATION
    return n * (250.0 + px * (12.0 + 2.0 * q))


def _solve_flops(px):
    # about five V(2, 1) cycles of 40 operations a cell on grids that add up to 4/3
    return px * 5.0 * 40.0 * 4.0 / 3.0


def work(case):
    kind, c = case["kind"], case["c"]
    if kind == "serve":
        sizes = [s for s in SV.SIZES if s[0] <= case["wmax"]]
        b = f = 0.0
        for i in range(case["requests"]):
            w, h = sizes[i % len(sizes)]
            b += _gaussian_bytes(case["n"], 2 * c) + 4.0 * c * w * h
            f += _composite_flops(case["n"], w, 2 * c) + _solve_flops(c * w * h)
        return {"bytes": b, "flops": f}
    px = float(c * case["w"] * case["h"])
    q = c if case.get("attr") == "laplacian" else 2 * c
    if kind == "project":
        return {"bytes": 4.0 * case["n"] * (11 + q + 2 + 3 + 1 + 4), "flops": 250.0 * case["n"]}
    if kind == "poisson":
        return {"bytes": px * 12.0, "flops": px * 4.0 + _solve_flops(px)}
    if kind == "rho":
        return {"bytes": px * 8.0, "flops": _solve_flops(px)}
    b, f = _gaussian_bytes(case["n"], q), _composite_flops(case["n"], case["w"], q)
    if kind == "maps":
        return {"bytes": b + px * 4.0 * (q // c), "flops": f}
    if kind == "view":
        return {"bytes": b + px * 4.0, "flops": f + _solve_flops(px)}
    # image and target and the image's gradient; the parameters once each way, their gradients out
    return {"bytes": 3.0 * b + px * 12.0, "flops": 3.5 * f + 2.0 * _solve_flops(px)}


# ------------------------------------------------------------------ the same in 64 bits

def _divergence(maps):
    gx, gy = maps[:, 0], maps[:, 1]
    rho = torch.zeros_like(gx)
    rho[:, :, :-1] += gx[:, :, :-1]
    rho[:, :, 1:] -= gx[:, :, :-1]
    rho[:, :-1, :] += gy[:, :-1, :]
    rho[:, 1:, :] -= gy[:, :-1, :]
    return rho


def _neumann(rho, mean):
    """The zero-mean Neumann solution of L u = rho - mean(rho), plus the mean: the
    5-point Laplacian is diagonal in the Fourier modes of the even extension."""
    c, h, w = rho.shape
    ky = torch.arange(2 * h, device=rho.device, dtype=torch.float64)
    kx = torch.arange(w + 1, device=rho.device, dtype=torch.float64)
    lam = ((2.0 * torch.cos(math.pi * ky / h) - 2.0)[:, None]
           + (2.0 * torch.cos(math.pi * kx / w) - 2.0)[None, :])
    lam[0, 0] = 1.0
    out = torch.empty_like(rho)
    for k in range(c):
        e = torch.cat([rho[k], rho[k].flip(0)], 0)
        e = torch.cat([e, e.flip(1)], 1)
        f = torch.fft.rfft2(e) / lam
        f[0, 0] = 0.0
        u = torch.fft.irfft2(f, s=(2 * h, 2 * w))[:h, :w]
        out[k] = u - u.mean() + mean[k]
    return out


def _camera64(cam):
    w2c = torch.as_tensor(np.asarray(cam.world_to_cam, dtype=np.float32)).double().cuda()
    return w2c, [float(np.float32(v)) for v in (cam.fx, cam.fy, cam.cx, cam.cy, cam.near)]


def _project64(p, cam):
    """Centre, covariance, depth and visibility by the definitions; p: PARAMS -> float64."""
    w2c, (fx, fy, cx, cy, near) = _camera64(cam)
    q = p["quat"] / p["quat"].norm(dim=1, keepdim=True)
    a, b, c, d = q.unbind(1)
    rot = torch.stack([1 - 2 * (c * c + d * d), 2 * (b * c - a * d), 2 * (b * d + a * c),
                       2 * (b * c + a * d), 1 - 2 * (b * b + d * d), 2 * (c * d - a * b),
                       2 * (b * d - a * c), 2 * (c * d + a * b), 1 - 2 * (b * b + c * c)], 1).view(-1, 3, 3)
    m = rot * p["scale"][:, None, :]
    t = p["mean"] @ w2c[:, :3].T + w2c[:, 3]
    z = t[:, 2]
    front = z > near
    zs = torch.where(front, z, torch.ones_like(z))
    zero = torch.zeros_like(z)
    jac = torch.stack([fx / zs, zero, -fx * t[:, 0] / zs ** 2,
                       zero, fy / zs, -fy * t[:, 1] / zs ** 2], 1).view(-1, 2, 3)
    g = jac @ w2c[:, :3] @ m
    cov = g @ g.transpose(1, 2)
    sxx, sxy, syy = cov[:, 0, 0] + DILATION, cov[:, 0, 1], cov[:, 1, 1] + DILATION
    u, v = fx * t[:, 0] / zs + cx, fy * t[:, 1] / zs + cy
    amin = float(np.float32(ALPHA_MIN))
    lev = torch.log((p["opacity"] / amin).clamp_min(1.0)).detach()
    # the footprint's half extents, a little wider so that no reachable pixel is left out
    rx = (torch.sqrt(sxx.detach() * lev) * 1.0001 + 1e-3)
    ry = (torch.sqrt(syy.detach() * lev) * 1.0001 + 1e-3)
    tx, ty = -(-cam.width // TILE), -(-cam.height // TILE)
    ud, vd = u.detach(), v.detach()
    x0 = torch.floor((ud - rx - 0.5) / TILE).clamp(0, tx)
    x1 = (torch.floor((ud + rx - 0.5) / TILE) + 1).clamp(0, tx)
    y0 = torch.floor((vd - ry - 0.5) / TILE).clamp(0, ty)
    y1 = (torch.floor((vd + ry - 0.5) / TILE) + 1).clamp(0, ty)
    vis = front & (p["opacity"] >= amin) & (x1 > x0) & (y1 > y0)
    return {"u": u, "v": v, "sxx": sxx, "sxy": sxy, "syy": syy, "z": z, "vis": vis,
            "box": torch.stack([x0, y0, x1, y1], 1).long()}


def _tile_lists(pr, cam):
    """Per tile its Gaussians in depth order (ties by index): (order of pairs, start of
    each tile's run, its length)."""
    tx, ty = -(-cam.width // TILE), -(-cam.height // TILE)
    idx = torch.nonzero(pr["vis"])[:, 0]
    idx = idx[torch.sort(pr["z"].detach()[idx], stable=True).indices]
    box = pr["box"][idx]
    nx, ny = box[:, 2] - box[:, 0], box[:, 3] - box[:, 1]
    cnt = nx * ny
    who = torch.repeat_interleave(torch.arange(len(idx), device=idx.device), cnt)
    k = torch.arange(len(who), device=idx.device) - torch.repeat_interleave(torch.cumsum(cnt, 0) - cnt, cnt)
    tile = (box[who, 1] + k // nx[who]) * tx + box[who, 0] + k % nx[who]
    tile, perm = torch.sort(tile, stable=True)
    num = torch.bincount(tile, minlength=tx * ty)
    return idx[who[perm]], torch.cumsum(num, 0) - num, num


def _composite64(p2, attr, cam, lists, d_maps=None):
    """Front-to-back composite of attr [n][q] over the image. p2: u, v, conic a, b, c,
    opacity. With d_maps, its gradient is accumulated into the leaves instead."""
    pairs, start, num = lists
    dev, q = attr.device, attr.shape[1]
    tx, ty = -(-cam.width // TILE), -(-cam.height // TILE)
    amin, amax, tmin = (float(np.float32(v)) for v in (ALPHA_MIN, ALPHA_MAX, T_MIN))
    canvas = torch.zeros((q, ty * TILE, tx * TILE), dtype=torch.float64, device=dev)
    if d_maps is not None:
        canvas[:, :cam.height, :cam.width] = d_maps
    blocks = canvas.view(q, ty, TILE, tx, TILE)
    off = torch.arange(TILE * TILE, device=dev)
    oy, ox = off // TILE, off % TILE
    by_len = torch.sort(num, descending=True).indices
    lens = num[by_len].tolist()
    budget = (4 if d_maps is not None else 12) << 20  # pixel-splat pairs held at once
    i, total = 0, sum(1 for v in lens if v > 0)
    while i < total:
        kmax = lens[i]
        take = max(1, min(total - i, budget // (kmax * TILE * TILE)))
        tiles = by_len[i:i + take]
        i += take
        slot = torch.arange(kmax, device=dev)[None, :]
        ok = slot < num[tiles][:, None]
        g = pairs[(start[tiles][:, None] + slot).clamp_max(len(pairs) - 1)]
        yy, xx = tiles // tx, tiles % tx
        px = (xx[:, None] * TILE + ox[None, :]).double()[:, None, :] + 0.5
        py = (yy[:, None] * TILE + oy[None, :]).double()[:, None, :] + 0.5
        dx, dy = px - p2["u"][g][:, :, None], py - p2["v"][g][:, :, None]
        power = (p2["a"][g][:, :, None] * dx * dx + p2["c"][g][:, :, None] * dy * dy
                 + 2.0 * p2["b"][g][:, :, None] * dx * dy)
        raw = p2["opacity"][g][:, :, None] * torch.exp(-power)
        al = torch.where(raw < amax, raw, torch.full_like(raw, amax))
        al = torch.where(ok[:, :, None] & (al >= amin), al, torch.zeros_like(al))
        after = torch.cumprod(1.0 - al, 1)
        before = torch.cat([torch.ones_like(after[:, :1]), after[:, :-1]], 1)
        wgt = torch.where(before.detach() >= tmin, al * before, torch.zeros_like(al))
        acc = torch.einsum("tkp,tkq->tqp", wgt, attr[g])
        if d_maps is None:
            blocks[:, yy, :, xx, :] = acc.view(-1, q, TILE, TILE)
        else:
            torch.autograd.backward(acc, blocks[:, yy, :, xx, :].reshape(-1, q, TILE * TILE))
    return canvas[:, :cam.height, :cam.width]


def _conic(pr, p):
    det = pr["sxx"] * pr["syy"] - pr["sxy"] ** 2
    return {"u": pr["u"], "v": pr["v"], "a": pr["syy"] / det, "b": -pr["sxy"] / det,
            "c": pr["sxx"] / det, "opacity": p["opacity"]}


def _params64(sc):
    return {k: torch.as_tensor(np.asarray(getattr(sc, k))).double().cuda() for k in PARAMS}


def _maps64(p, cam):
    pr = _project64(p, cam)
    n, q = p["grad"].shape[0], p["grad"][0].numel()
    return _composite64(_conic(pr, p), p["grad"].reshape(n, q), cam, _tile_lists(pr, cam))


def _image64(maps, laplacian, mean, c):
    h, w = maps.shape[-2:]
    return _neumann(maps.reshape(c, h, w) if laplacian else _divergence(maps.reshape(c, 2, h, w)), mean)


def exact(case, seed):
    kind, c = case["kind"], case["c"]
    mean = [float(np.float32(m)) for m in _means(c)]
    if kind == "poisson":
        maps, mask = _poisson_inputs(case, seed)
        if mask is not None:
            on = mask.repeat_interleave(TILE, 0).repeat_interleave(TILE, 1)[:case["h"], :case["w"]]
            maps = maps * on
        return _neumann(_divergence(maps.double()), mean)
    if kind == "rho":
        rho, t = _rho_input(case, seed), case.get("threshold") or 0.0
        return _neumann(torch.where(rho.abs() >= t, rho, torch.zeros_like(rho)).double(), mean)
    sc, cam = _scene(case, seed)
    p = _params64(sc)
    lap = case.get("attr") == "laplacian"
    if kind == "serve":
        return [_image64(_maps64(p, r.cam), lap, mean, c) for r in _requests(case, seed)]
    if kind == "project":
        pr = _project64(p, cam)
        keep = lambda *v: torch.stack(v, 1) * pr["vis"][:, None]  # noqa: E731
        return {"mean2d": keep(pr["u"], pr["v"]), "cov2d": keep(pr["sxx"], pr["sxy"], pr["syy"]),
                "depth": pr["z"] * pr["vis"], "rect": None}
    if kind == "maps":
        m = _maps64(p, cam)
        return m if lap else m.reshape(c, 2, case["h"], case["w"])
    if kind == "view":
        return _image64(_maps64(p, cam), lap, mean, c)
    # train: the image, d image through the solve's and the divergence's transposes, then
    # autograd through the composite (tile by tile) and the projection
    for v in p.values():
        v.requires_grad_(True)
    pr = _project64(p, cam)
    q = p["grad"][0].numel()
    p2 = _conic(pr, p)
    leaf = {k: v.detach().requires_grad_(True) for k, v in p2.items()}
    attr = p["grad"].detach().reshape(-1, q).requires_grad_(True)
    lists = _tile_lists(pr, cam)
    with torch.no_grad():
        img = _image64(_composite64({k: v.detach() for k, v in leaf.items()}, attr.detach(), cam, lists),
                       lap, mean, c)
        d_img = 2.0 * (img - _photo(c, case["h"], case["w"], seed + 2).double()) / img.numel()
        d_rho = _neumann(d_img, [0.0] * c)
        d_maps = d_rho if lap else -_gradient_maps(d_rho)
    _composite64(leaf, attr, cam, lists, d_maps.reshape(q, case["h"], case["w"]))
    keys = ("u", "v", "a", "b", "c")
    shape = ("mean", "scale", "quat")
    got = torch.autograd.grad([p2[k] for k in keys], [p[k] for k in shape],
                              [leaf[k].grad * pr["vis"] for k in keys])
    out = {"d_" + k: v for k, v in zip(shape, got)}
    out["d_opacity"] = leaf["opacity"].grad
    out["d_grad"] = attr.grad.reshape(p["grad"].shape)
    out["image"] = img
    return out
