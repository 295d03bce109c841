"""Timed cases of the renderer: the calls a program makes through ``raster``, on synthetic scenes.

A case names an operation, a scene recipe (the distributions of ``scenes.py``, drawn here on
the GPU from the case's seed) and sizes.  Operations:

  frame         projection, binning and forward of one view (a viewer's frame)
  project       projection of every Gaussian into a batch of views
  project_grad  the projection's backward over a batch of views
  sh            spherical-harmonics colour of a batch of views and its backward
  bin           complete per-tile lists of one view
  bin_views     truncated per-tile lists of a batch of views
  render        differentiable render of one view and its backward (``raster.render``)
  step          a training step of one view: projection, SH colour, binning, render, L2 loss,
                backward to the 3D parameters
  step_views    projection, truncated lists, render, L2 loss gradient and render backward of a
                batch of views, replayed as the plan's CUDA graph (the benchmark's step)

Plans: "default" is ``raster.Plan()``; "pixel" and "segments" are the knobs the autotuner keeps
on the dense frames (pixel-wise items, 4 rows per lane) and on frames with a few very long
lists (Gaussian-wise items of 8 pixels for lists past 4096 entries).
"""
from __future__ import annotations

import math

import torch

from paper_2412_17378_gb300 import raster, scenes

DEV = "cuda"
TILE = 16
NEVER = 2147483647
LARGEST = -2.5

PLANS = {
    "default": {},
    "pixel": dict(pixel_rows=4, heavy_threshold=NEVER),
    "segments": dict(pixel_rows=4, heavy_threshold=4096, gw_pixels=8),
}

# recipe: log-scale mean and deviation, then evaluated pairs per pixel, tiles per Gaussian and
# kept entries per record of a truncated list (rounded measurements, for work() alone)
RECIPES = {
    "box": (-3.5, 0.5, 40, 4, 4),
    "clustered": (-4.0, 0.7, 220, 60, 20),
    "early": (-2.0, 0.5, 350, 600, 30),
    "late": (-5.0, 0.5, 120, 5, 4),
    "clusters3": (-4.5, 1.0, 290, 90, 6),
    "veil": (-4.0, 0.7, 900, 40, 20),
}


def listed():
    return [
        # the smallest frame of the workloads: latency of the launches and of the one read-back
        dict(name="frame_256_10k", op="frame", scene="box", n=10_000, w=256, h=256, plan="default"),
        # an ordinary viewer's frame: an imbalanced full-HD view, tuned knobs
        dict(name="frame_1080p_600k", op="frame", scene="clustered", n=600_000, w=1920, h=1080, plan="pixel"),
        # projection of a batch of training views, and its backward
        dict(name="project_8x1m", op="project", scene="clustered", n=1_000_000, w=1280, h=720, views=8, plan="pixel"),
        dict(name="project_grad_4x1m", op="project_grad", scene="clustered", n=1_000_003, w=1280, h=720, views=4,
             plan="pixel"),
        # view-dependent colour (degree 3) of one training view, forward and backward
        dict(name="sh_degree3_1m", op="sh", scene="clustered", n=1_000_000, w=1920, h=1080, views=1, degree=3,
             plan="pixel"),
        # complete lists of an imbalanced full-HD view
        dict(name="bin_1080p_1m", op="bin", scene="clustered", n=1_000_000, w=1920, h=1080, plan="pixel"),
        # truncated lists of a batch of views of mixed sizes
        dict(name="bin_views_16x500k", op="bin_views", scene="clustered", n=500_000, w=1920, h=1080, views=16,
             plan="pixel"),
        # an early training stage: few large faint Gaussians; depth and alpha are supervised too
        dict(name="render_720p_early", op="render", scene="early", n=100_000, w=1280, h=720, plan="pixel", extra=True),
        # an imbalanced full-HD view under the plan's defaults
        dict(name="render_1080p_default", op="render", scene="clustered", n=300_000, w=1920, h=1080, plan="default",
             extra=False),
        # a few ultra-heavy tiles under the knobs the autotuner keeps for them
        dict(name="render_1080p_veil", op="render", scene="veil", n=300_000, w=1920, h=1080, plan="segments",
             extra=False),
        # a late training stage (many small opaque Gaussians): the whole step of one view, with
        # an image whose sides are no multiple of the tile
        dict(name="step_720p_late", op="step", scene="late", n=3_000_000, w=1279, h=717, degree=3, plan="default"),
        # the whole step of a 3840x2160 view and eight 1920x1080 views
        dict(name="step_9views_4m", op="step_views", scene="clusters3", n=4_000_000, w=3840, h=2160, views=9,
             plan="pixel"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["frame", "frame", "project", "project_grad", "sh", "bin", "bin_views", "render", "render", "step",
                     "step_views"])
    if op in ("project", "project_grad", "sh"):
        views = rng.randint(1, 12)
        c = dict(op=op, scene=rng.choice(["clustered", "late", "clusters3"]), n=_log_int(rng, 2_000, 4_000_000 // views),
                 w=rng.randint(200, 1920), h=rng.randint(200, 1080), views=views, plan="pixel")
        if op == "sh":
            c["degree"] = rng.choice([1, 2, 3, 3])
        return c
    if op in ("bin_views", "step_views"):
        views = rng.randint(2, 10)
        return dict(op=op, scene=rng.choice(["clustered", "late", "clusters3"]), n=_log_int(rng, 5_000, 500_000),
                    w=rng.randint(200, 1920), h=rng.randint(200, 1080), views=views, plan="pixel")
    w = _log_int(rng, 64, 1920)
    scene = rng.choice(["box", "clustered", "clustered", "early", "late"])
    most = dict(box=200_000, clustered=600_000, early=60_000, late=2_000_000)[scene]
    c = dict(op=op, scene=scene, n=_log_int(rng, 500, most), w=w, h=max(48, int(w * rng.uniform(0.5, 1.0))),
             plan=rng.choice(["default", "pixel"]))
    if op == "render":
        c["extra"] = rng.random() < 0.5
    if op == "step":
        c["degree"] = rng.choice([0, 1, 3])
    return c


# ---- scenes (the distributions of scenes.py, drawn on the GPU) -------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _u(g, lo, hi, *shape):
    return torch.rand(*shape, generator=g, device=DEV) * (hi - lo) + lo


def _n(g, mean, dev, *shape):
    return torch.randn(*shape, generator=g, device=DEV) * dev + mean


def _frustum(g, n, W, H, z_lo=2.0, z_hi=6.0, window=None):
    """Points whose projections are uniform over the identity camera's image (or a window of it)."""
    u0, u1, v0, v1 = window or (0.0, W, 0.0, H)
    z = _u(g, z_lo, z_hi, n)
    x = (_u(g, u0, u1, n) - (W - 1) / 2) / W * z
    y = (_u(g, v0, v1, n) - (H - 1) / 2) / W * z
    return torch.stack([x, y, z], 1)


def _cluster(g, n, W, H, pu, pv, z, sigma):
    c = torch.tensor([(pu * W - (W - 1) / 2) / W * z, (pv * H - (H - 1) / 2) / W * z, z], device=DEV)
    return c + sigma * _n(g, 0.0, 1.0, n, 3)


def _gaussians(case, g):
    """means3D, log_scales, quats, opacities, colors of the case's scene."""
    n, W, H, scene = case["n"], case["w"], case["h"], case["scene"]
    mu, dev = RECIPES[scene][:2]
    ls = _n(g, mu, dev, n, 3)
    op = torch.sigmoid(_n(g, 0.0, 1.5, n))
    if scene == "box":
        means = torch.stack([_u(g, -1, 1, n), _u(g, -1, 1, n), _u(g, 2, 6, n)], 1)
        op = torch.sigmoid(_n(g, 0.0, 1.0, n))
    elif scene == "clustered":
        nc = int(0.8 * n)
        means = torch.cat([_cluster(g, nc, W, H, 0.3, 0.6, 4.0, 0.189), _frustum(g, n - nc, W, H)])
    elif scene == "early":
        means, op = _frustum(g, n, W, H), _u(g, 0.05, 0.3, n)
    elif scene == "late":
        means, op = _frustum(g, n, W, H), _u(g, 0.5, 1.0, n)
    elif scene == "clusters3":
        n1, n2, n3 = int(0.6 * n), int(0.2 * n), int(0.1 * n)
        means = torch.cat([_cluster(g, n1, W, H, 0.3, 0.6, 4.0, 0.25), _cluster(g, n2, W, H, 0.7, 0.35, 3.5, 0.2),
                           _cluster(g, n3, W, H, 0.55, 0.5, 5.0, 0.15), _frustum(g, n - n1 - n2 - n3, W, H)])
        op = torch.sigmoid(_n(g, 0.5, 1.5, n))
        ls.clamp_(max=LARGEST)  # as training prunes the largest Gaussians
    else:  # a veil of faint Gaussians over 48 x 48 pixels, in front of a clustered scene
        nv = n // 3
        nb = n - nv
        nc = int(0.8 * nb)
        u, v = 0.62 * W, 0.4 * H
        means = torch.cat([_cluster(g, nc, W, H, 0.3, 0.6, 4.0, 0.189), _frustum(g, nb - nc, W, H),
                           _frustum(g, nv, W, H, 1.0, 1.9, (u - 24, u + 24, v - 24, v + 24))])
        ls[nb:] = _n(g, -5.6, 0.15, nv, 3)
        op[nb:] = _u(g, 0.001, 0.0045, nv)
    q = _n(g, 0.0, 1.0, n, 4)
    q = q / q.norm(dim=1, keepdim=True)
    return [t.contiguous() for t in (means, ls, q, op, _u(g, 0, 1, n, 3))]


def _cameras(case):
    V, W, H = case.get("views", 1), case["w"], case["h"]
    if V == 1:
        return [scenes.camera(W, H)]
    if case["op"] == "step_views" and W == 3840:  # one large view and the others at half its sides
        return [scenes.camera(W, H)] + scenes.arc_cameras([(W // 2, H // 2)] * (V - 1))
    third = lambda k: (W * k // 3, H * k // 3)
    return scenes.arc_cameras([third(1) if k % 4 == 0 else third(3) if k % 4 == 2 else third(2) for k in range(V)])


# ---- the projection and the render in plain torch (inputs in 32 bits, exact values in 64) ----

def _project(means, ls, quats, cam):
    """Projection of the Gaussians into one view: means2D, conic (a, b, c), depth, radius (0: not seen)."""
    dt = means.dtype
    V = torch.as_tensor(cam["viewmat"], dtype=dt, device=DEV)
    fx, fy, W, H = cam["fx"], cam["fy"], cam["W"], cam["H"]
    p = means @ V[:3, :3].T + V[:3, 3]
    z = p[:, 2]
    seen = z > cam["near"]
    zs = torch.where(seen, z, torch.ones_like(z))
    w, x, y, k = (quats / quats.norm(dim=1, keepdim=True)).unbind(1)
    R = torch.stack([1 - 2 * (y * y + k * k), 2 * (x * y - w * k), 2 * (x * k + w * y),
                     2 * (x * y + w * k), 1 - 2 * (x * x + k * k), 2 * (y * k - w * x),
                     2 * (x * k - w * y), 2 * (y * k + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    M = R * ls.exp()[:, None, :]
    limx, limy = 1.3 * W / (2 * fx), 1.3 * H / (2 * fy)
    cx, cy = (p[:, 0] / zs).clamp(-limx, limx), (p[:, 1] / zs).clamp(-limy, limy)
    r0 = (fx / zs)[:, None] * (V[0, :3] - cx[:, None] * V[2, :3])
    r1 = (fy / zs)[:, None] * (V[1, :3] - cy[:, None] * V[2, :3])
    P0, P1 = (r0[:, :, None] * M).sum(1), (r1[:, :, None] * M).sum(1)
    A, B, C = (P0 * P0).sum(1) + cam["lowpass"], (P0 * P1).sum(1), (P1 * P1).sum(1) + cam["lowpass"]
    det = A * C - B * B
    m2 = torch.stack([fx * p[:, 0] / zs + cam["cx"], fy * p[:, 1] / zs + cam["cy"]], 1)
    conic = torch.stack([C / det, -B / det, A / det], 1)
    with torch.no_grad():
        lam = (A + C) / 2 + (((A - C) / 2) ** 2 + B * B).clamp_min(0.1).sqrt()
        r = torch.where(seen, (3 * lam.sqrt()).ceil(), torch.zeros_like(z))
        x0, x1, y0, y1 = _rect(m2, r, cam)
        r = torch.where((x1 > x0) & (y1 > y0), r, torch.zeros_like(r))
    s = seen[:, None]
    return torch.where(s, m2, torch.zeros_like(m2)), torch.where(s, conic, torch.zeros_like(conic)), z, r


def _rect(m2, r, cam):
    tx, ty = -(-cam["W"] // TILE), -(-cam["H"] // TILE)
    lo = lambda u, t: torch.floor((u - r) / TILE).clamp(0, t).long()
    hi = lambda u, t: torch.floor((u + (r + TILE - 1)) / TILE).clamp(0, t).long()
    return lo(m2[:, 0], tx), hi(m2[:, 0], tx), lo(m2[:, 1], ty), hi(m2[:, 1], ty)


def _lists(m2, r, depth, cam):
    """Every tile's Gaussians in depth order: (index list, first entry per tile, entries per tile)."""
    tx, ty = -(-cam["W"] // TILE), -(-cam["H"] // TILE)
    order = torch.sort(depth.float(), stable=True).indices
    order = order[r[order] > 0]
    x0, x1, y0, y1 = (t[order] for t in _rect(m2.float(), r.float(), cam))
    w = x1 - x0
    cnt = w * (y1 - y0)
    src = torch.repeat_interleave(torch.arange(order.numel(), device=DEV), cnt)
    k = torch.arange(src.numel(), device=DEV) - (torch.cumsum(cnt, 0) - cnt)[src]
    tile = ((y0[src] + k // w[src]) * tx + x0[src] + k % w[src]).int()
    by = torch.sort(tile, stable=True).indices
    n = torch.bincount(tile, minlength=tx * ty)
    return order[src[by]], torch.cumsum(n, 0) - n, n


def _walk(m2, conic, op, feat, lists, cam, grad=None, chunk=16):
    """The blend in 64 bits, `chunk` entries of every pixel's list at a time: the features (colour
    and depth) and the transmittance left [pixels].  With `grad` = (gradient of the blended
    features [pixels, F], total per pixel) the gradients of (m2, conic, op, feat) instead."""
    idx, first, count = lists
    W, H = cam["W"], cam["H"]
    tx = -(-W // TILE)
    py, px = torch.meshgrid(torch.arange(H, device=DEV), torch.arange(W, device=DEV), indexing="ij")
    px, py = px.reshape(-1), py.reshape(-1)
    tile = (py // TILE) * tx + px // TILE
    F = feat.shape[1]
    T = torch.ones(W * H, dtype=torch.float64, device=DEV)
    acc = torch.zeros(W * H, F, dtype=torch.float64, device=DEV)
    run = torch.zeros(W * H, dtype=torch.float64, device=DEV)
    out = None if grad is None else [torch.zeros(t.shape, dtype=torch.float64, device=DEV) for t in (m2, conic, op, feat)]
    live, pos = torch.arange(W * H, device=DEV), 0
    step = torch.arange(chunk, device=DEV)
    while live.numel():
        live = live[count[tile[live]] > pos]
        parts = []
        for a in live.split(1 << 19):
            e = first[tile[a]][:, None] + pos + step
            ok = pos + step < count[tile[a]][:, None]
            g = idx[torch.where(ok, e, 0)]
            dx, dy = m2[g, 0] - px[a][:, None], m2[g, 1] - py[a][:, None]
            ca, cb, cc = conic[g, 0], conic[g, 1], conic[g, 2]
            power = -0.5 * (ca * dx * dx + cc * dy * dy) - cb * dx * dy
            oG = op[g] * power.exp()
            ok &= (power <= 0) & (oG >= 1 / 255)
            al = torch.where(ok, oG.clamp_max(0.99), 0.0)
            after = T[a][:, None] * torch.cumprod(1 - al, 1)
            before = torch.cat([T[a][:, None], after[:, :-1]], 1)
            go = after >= 1e-4  # a prefix: the first entry below stops the pixel
            ok &= go
            w = torch.where(ok, al * before, 0.0)
            if grad is None:
                acc[a] += (w[:, :, None] * feat[g]).sum(1)
            else:
                up, total = grad
                dot = (feat[g] * up[a][:, None, :]).sum(2)
                done = run[a][:, None] + torch.cumsum(w * dot, 1)
                da = torch.where(ok, before * dot - (total[a][:, None] - done) / (1 - al), 0.0)
                run[a] = done[:, -1]
                q = torch.nonzero(ok, as_tuple=True)
                gq, wq = g[q], w[q]
                out[3].index_add_(0, gq, wq[:, None] * up[a][q[0]])
                dp = torch.where(oG[q] > 0.99, 0.0, oG[q] * da[q])
                dxq, dyq = dx[q], dy[q]
                out[2].index_add_(0, gq, dp / op[gq])
                out[0].index_add_(0, gq, torch.stack([-dp * (ca[q] * dxq + cb[q] * dyq),
                                                      -dp * (cc[q] * dyq + cb[q] * dxq)], 1))
                out[1].index_add_(0, gq, torch.stack([-0.5 * dp * dxq * dxq, -dp * dxq * dyq, -0.5 * dp * dyq * dyq], 1))
            left = torch.where(go, after, 2.0).amin(1)  # the last transmittance kept
            T[a] = torch.where(left > 1.5, T[a], left)
            parts.append(a[go[:, -1]])
        live = torch.cat(parts) if parts else live[:0]
        pos += chunk
    return out if grad is not None else (acc, T)


def _render64(m2, conic, op, colors, depth, lists, cam):
    """color [3,H,W], depth [H,W], alpha [H,W]."""
    acc, T = _walk(m2, conic, op, torch.cat([colors, depth[:, None]], 1), lists, cam)
    H, W = cam["H"], cam["W"]
    img = acc.T.reshape(4, H, W)
    return img[:3].contiguous(), img[3].contiguous(), (1 - T).reshape(H, W)


def _render64_grad(m2, conic, op, colors, depth, lists, cam, img, up):
    """Gradients of sum(up * image) with respect to (m2, conic, op, colors, depth); up: color, depth, alpha."""
    n = cam["W"] * cam["H"]
    flat = lambda t, k: t.double().reshape(k, n).T
    feat = torch.cat([colors, depth[:, None], torch.ones_like(depth)[:, None]], 1)  # alpha blends a one
    u = torch.cat([flat(up[0], 3), flat(up[1], 1), flat(up[2], 1)], 1)
    total = (u * torch.cat([flat(img[0], 3), flat(img[1], 1), flat(img[2], 1)], 1)).sum(1)
    gm, gc, go, gf = _walk(m2, conic, op, feat, lists, cam, grad=(u, total))
    return gm, gc, go, gf[:, :3].contiguous(), gf[:, 3].contiguous()


def _sh64(sh, means, centre, degree):
    d = means - centre
    x, y, z = (d / d.norm(dim=1, keepdim=True)).unbind(1)
    xx, yy, zz, s = x * x, y * y, z * z, math.sqrt
    pi = math.pi
    Y = [torch.full_like(x, 0.5 / s(pi))]
    if degree > 0:
        Y += [-s(3 / (4 * pi)) * y, s(3 / (4 * pi)) * z, -s(3 / (4 * pi)) * x]
    if degree > 1:
        a = s(15 / pi) / 2
        Y += [a * x * y, -a * y * z, s(5 / pi) / 4 * (2 * zz - xx - yy), -a * x * z, a / 2 * (xx - yy)]
    if degree > 2:
        a, b, c = s(35 / (2 * pi)) / 4, s(105 / pi) / 2, s(21 / (2 * pi)) / 4
        Y += [-a * y * (3 * xx - yy), b * x * y * z, -c * y * (4 * zz - xx - yy),
              s(7 / pi) / 4 * z * (2 * zz - 3 * xx - 3 * yy), -c * x * (4 * zz - xx - yy), b / 2 * z * (xx - yy),
              -a * x * (xx - 3 * yy)]
    return ((torch.stack(Y, 1)[:, :, None] * sh[:, :len(Y)]).sum(1) + 0.5).clamp_min(0)


def _centre(cam):
    V = torch.as_tensor(cam["viewmat"], dtype=torch.float64, device=DEV)
    return -V[:3, :3].T @ V[:3, 3]


# ---- inputs ----------------------------------------------------------------------------------

def _inputs(case, seed):
    """What the caller has in hand: parameters, cameras, upstream gradients or targets."""
    g = _gen(seed)
    op, n = case["op"], case["n"]
    m3, ls, q, o, col = _gaussians(case, g)
    cams = _cameras(case)
    cam = cams[0]
    W, H = cam["W"], cam["H"]
    x = dict(m3=m3, ls=ls, q=q, op=o, col=col, cams=cams, cam=cam, W=W, H=H)
    if op in ("render", "bin"):
        m2, conic, z, r = _project(m3, ls, q, cam)
        x.update(m2=m2.contiguous(), co=torch.cat([conic, o[:, None]], 1).contiguous(), z=z.contiguous(),
                 r=r.int().contiguous())
    if op in ("bin_views", "project_grad"):
        per = [_project(m3, ls, q, c) for c in cams]
        x.update(m2=torch.cat([p[0] for p in per]), z=torch.cat([p[2] for p in per]),
                 co=torch.cat([torch.cat([p[1], o[:, None]], 1) for p in per]),
                 r=torch.cat([p[3] for p in per]).int())
    if op == "project_grad":
        R = n * len(cams)
        x.update(g_m2=_n(g, 0, 1, R, 2), g_conic=_n(g, 0, 1, R, 3), g_z=_n(g, 0, 1, R))
    if op == "render":
        x.update(g_color=_n(g, 0, 1, 3, H, W), g_depth=_n(g, 0, 0.1, H, W), g_alpha=_n(g, 0, 0.1, H, W))
    if op in ("sh", "step"):
        x["sh"] = _n(g, 0, 0.3, n, (case["degree"] + 1) ** 2, 3)
        x["g_rgb"] = _n(g, 0, 1, n * len(cams), 3) if op == "sh" else None
    if op == "step":
        x["target"] = _u(g, 0, 1, 3, H, W)
    if op == "step_views":
        x["targets"] = [_u(g, 0, 1, 3, c["H"], c["W"]) for c in cams]
    return x


def _capacity(case):
    """Slots of the caller's point-list buffer: above every list these scenes give at these sizes."""
    per = dict(box=16, clustered=110, early=1000, late=24, clusters3=110)[case["scene"]]
    records = case["n"] * case.get("views", 1)
    return min(int(records * (16 + per * (case["w"] / 1280) ** 2)), 500_000_000)


def prepare(case, seed):
    s = _inputs(case, seed)
    op = case["op"]
    s["case"] = case
    s["plan"] = plan = raster.Plan(**PLANS[case["plan"]])
    s["list"] = None  # the point-list buffer, kept from the first call on
    if op in ("bin", "bin_views"):
        s["list"] = torch.zeros(_capacity(case), dtype=torch.int32, device=DEV)
    if op == "render":
        s["binning"] = raster.bin_and_sort(plan, s["m2"], s["r"], s["z"], s["W"], s["H"])
    if op == "render":
        s["leaves"] = [s[k].requires_grad_(True) for k in ("m2", "co", "col", "z")]
    if op == "step":
        s["leaves"] = [s[k].requires_grad_(True) for k in ("m3", "ls", "q", "op", "sh")]
    if op == "sh":
        s["leaves"] = [s[k].requires_grad_(True) for k in ("sh", "m3")]
    if op == "step_views":
        _capture(s)
    return s


def _capture(s):
    """Sizes the point list with one synchronous pass, runs the step once and captures it."""
    plan, cams = s["plan"], s["cams"]
    pre = raster.preprocess_batched(plan, s["m3"], s["ls"], s["q"], s["op"], cams)
    pl, rg, K = raster.bin_and_sort_batched(plan, pre["means2D"], pre["radii"], pre["depths"], cams,
                                            conic_opacity=pre["conic_opacity"],
                                            point_list=torch.empty(8 * pre["depths"].numel(), dtype=torch.int32, device=DEV))
    pl = torch.empty(int(1.2 * K) + 1024, dtype=torch.int32, device=DEV)
    s.update(pre=pre, list=pl, ranges=rg, outs=raster.alloc_view_outputs(cams, DEV),
             g_img=[torch.empty_like(t) for t in s["targets"]], grads=None)

    def step():
        raster.preprocess_batched(plan, s["m3"], s["ls"], s["q"], s["op"], cams, out=pre)
        raster.bin_and_sort_batched(plan, pre["means2D"], pre["radii"], pre["depths"], cams, point_list=pl, ranges=rg,
                                    no_sync=True, conic_opacity=pre["conic_opacity"])
        raster.render_forward_batched(plan, pre["means2D"], pre["conic_opacity"], s["col"], pre["depths"], pl, pl.numel(),
                                      rg, cams, outs=s["outs"])
        for o, t, d in zip(s["outs"], s["targets"], s["g_img"]):
            torch.sub(o["color"], t, out=d)
        s["grads"] = raster.render_backward_batched(
            plan, pre["means2D"], pre["conic_opacity"], s["col"], pre["depths"], pl, pl.numel(), rg, cams, s["outs"],
            [dict(color=d) for d in s["g_img"]], out=s["grads"])

    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        step()
        torch.cuda.synchronize()
        raster.graph_begin(plan)
        step()
        raster.graph_end(plan)
    torch.cuda.current_stream().wait_stream(side)


# ---- one pass --------------------------------------------------------------------------------

def run(s):
    case, plan = s["case"], s["plan"]
    op, W, H = case["op"], s["W"], s["H"]
    if op == "frame":
        pre = raster.preprocess(plan, s["m3"], s["ls"], s["q"], s["op"], s["cam"])
        s["list"], ranges, K = raster.bin_and_sort(plan, pre["means2D"], pre["radii"], pre["depths"], W, H,
                                                   point_list=s["list"])
        img = raster.render_forward(plan, pre["means2D"], pre["conic_opacity"], s["col"], pre["depths"], s["list"], K,
                                    ranges, W, H)
        return dict(pre=pre, img=img)
    if op == "project":
        return raster.preprocess_batched(plan, s["m3"], s["ls"], s["q"], s["op"], s["cams"])
    if op == "project_grad":
        return raster.preprocess_backward_batched(plan, s["m3"], s["ls"], s["q"], s["cams"], s["r"], s["g_m2"],
                                                  s["g_conic"], s["g_z"])
    if op == "sh":
        rgb = raster.SHFunction.apply(s["sh"], s["m3"], plan, s["cams"], case["degree"])
        return [rgb, *torch.autograd.grad(rgb, s["leaves"], s["g_rgb"])]
    if op == "bin":
        s["list"], ranges, K = raster.bin_and_sort(plan, s["m2"], s["r"], s["z"], W, H, point_list=s["list"])
        return [s["list"], ranges, K]
    if op == "bin_views":
        s["list"], ranges, K = raster.bin_and_sort_batched(plan, s["m2"], s["r"], s["z"], s["cams"],
                                                           point_list=s["list"], conic_opacity=s["co"])
        return [s["list"], ranges, K]
    if op == "render":
        img = raster.render(plan, s["m2"], s["co"], s["col"], s["z"], s["binning"], W, H)
        ups = (s["g_color"], s["g_depth"], s["g_alpha"])
        k = 3 if case["extra"] else 1
        return [*img, *torch.autograd.grad(img[:k], s["leaves"], ups[:k])]
    if op == "step":
        for t in s["leaves"]:
            t.grad = None
        m2, co, z, radii = raster.PreprocessFunction.apply(s["m3"], s["ls"], s["q"], s["op"], plan, s["cam"], (TILE, TILE))
        colors = raster.SHFunction.apply(s["sh"], s["m3"], plan, s["cams"], case["degree"])
        binning = raster.bin_and_sort(plan, m2.detach(), radii, z.detach(), W, H, point_list=s["list"])
        s["list"] = binning[0]
        color, _, _ = raster.render(plan, m2, co, colors, z, binning, W, H)
        loss = 0.5 * ((color - s["target"]) ** 2).sum()
        loss.backward()
        return [color, loss, *[t.grad for t in s["leaves"]]]
    raster.graph_launch(plan)
    return dict(color=[o["color"] for o in s["outs"]], T=[o["final_T"] for o in s["outs"]], grads=s["grads"])


# ---- work and exact values -------------------------------------------------------------------

def work(case):
    """Bytes and flops a pass cannot do without: inputs read once, outputs written once; per
    evaluated pair 8 flops forward, and per blended one (about a third) 7 forward; backward 9 and 18."""
    n, V, op = case["n"], case.get("views", 1), case["op"]
    cams = _cameras(case)
    px = sum(c["W"] * c["H"] for c in cams)
    _, _, pairs, tiles, kept = RECIPES[case["scene"]]
    entries = n * tiles * min(1.0, case["w"] / 1280) ** 2  # of one view's complete lists
    fwd, bwd = px * pairs * (8 + 7 / 3), px * pairs * (9 + 18 / 3)
    k = (case.get("degree", 0) + 1) ** 2
    project = dict(bytes=44 * n + 36 * n * V, flops=150 * n * V)
    project_grad = dict(bytes=80 * n + 28 * n * V, flops=300 * n * V)
    lists = dict(bytes=12 * n + 4 * entries, flops=0)
    image = dict(bytes=48 * n + 4 * entries + 28 * px, flops=fwd)
    image_grad = dict(bytes=96 * n + 4 * entries + 20 * px, flops=bwd)
    sh = dict(bytes=(12 * k + 12) * 3 * n + 24 * n * V, flops=10 * k * n * V)
    vlists = dict(bytes=28 * n * V + 4 * kept * n * V, flops=0)
    vimage = dict(bytes=48 * n * V + 4 * kept * n * V + 28 * px, flops=fwd)
    vimage_grad = dict(bytes=96 * n * V + 4 * kept * n * V + 20 * px, flops=bwd)
    parts = dict(frame=[project, lists, image], project=[project], project_grad=[project_grad], sh=[sh],
                 bin=[lists], bin_views=[vlists], render=[image, image_grad],
                 step=[project, sh, lists, image, image_grad, project_grad],
                 step_views=[project, vlists, vimage, vimage_grad])[op]
    return {key: float(sum(p[key] for p in parts)) for key in ("bytes", "flops")}


def exact(case, seed):
    op = case["op"]
    if op in ("bin", "bin_views", "step_views") or case["scene"] == "veil":
        return None  # whole numbers; batches and very long lists take too long
    x = _inputs(case, seed)
    d = lambda *names: [x[k].double() for k in names]
    n, cams, cam, W, H = case["n"], x["cams"], x["cam"], x["W"], x["H"]
    if op == "project":
        per = [_project(*d("m3", "ls", "q"), c) for c in cams]
        return dict(means2D=torch.cat([p[0] for p in per]), depths=torch.cat([p[2] for p in per]), radii=None,
                    tiles_touched=None, conic_opacity=torch.cat([torch.cat([p[1], x["op"].double()[:, None]], 1) for p in per]))
    if op == "project_grad":
        leaves = [t.requires_grad_(True) for t in d("m3", "ls", "q")]
        total = [torch.zeros_like(t) for t in leaves]
        for v, c in enumerate(cams):
            m2, conic, z, _ = _project(*leaves, c)
            k = slice(v * n, (v + 1) * n)
            seen = (x["r"][k] > 0).double()[:, None]
            ups = [x["g_m2"][k].double() * seen, x["g_conic"][k].double() * seen, x["g_z"][k].double() * seen[:, 0]]
            for t, gr in zip(total, torch.autograd.grad([m2, conic, z], leaves, ups)):
                t += gr
        return dict(means3D=total[0], log_scales=total[1], quats=total[2])
    if op == "sh":
        sh, m3 = (t.requires_grad_(True) for t in d("sh", "m3"))
        rgb = torch.cat([_sh64(sh, m3, _centre(c), case["degree"]) for c in cams])
        return [rgb.detach(), *torch.autograd.grad(rgb, [sh, m3], x["g_rgb"].double())]
    if op == "render":
        m2, co, col, z = d("m2", "co", "col", "z")
        lists = _lists(x["m2"], x["r"], x["z"], cam)
        args = (m2, co[:, :3].contiguous(), co[:, 3].contiguous(), col, z, lists, cam)
        img = _render64(*args)
        k = 1.0 if case["extra"] else 0.0
        gm, gc, go, gcol, gz = _render64_grad(*args, img, (x["g_color"], k * x["g_depth"], k * x["g_alpha"]))
        return [*img, gm, torch.cat([gc, go[:, None]], 1), gcol, gz if case["extra"] else None]
    # frame, step: from the 3D parameters
    leaves = [t.requires_grad_(op == "step") for t in d("m3", "ls", "q", "op")]
    m2, conic, z, r = _project(*leaves[:3], cam)
    lists = _lists(m2.detach(), r, z.detach(), cam)
    if op == "frame":
        img = _render64(m2, conic, leaves[3], x["col"].double(), z, lists, cam)
        pre = dict(means2D=m2, conic_opacity=torch.cat([conic, leaves[3][:, None]], 1), depths=z, radii=None, tiles_touched=None)
        return dict(pre=pre, img=dict(color=img[0], depth=img[1], alpha=img[2], final_T=1 - img[2], n_contrib=None))
    sh = x["sh"].double().requires_grad_(True)
    colors = _sh64(sh, leaves[0], _centre(cam), case["degree"])
    args = tuple(t.detach() for t in (m2, conic, leaves[3], colors, z)) + (lists, cam)
    img = _render64(*args)
    diff = img[0] - x["target"].double()
    zero = torch.zeros(H, W, dtype=torch.float64, device=DEV)
    gm, gc, go, gcol, _ = _render64_grad(*args, img, (diff, zero, zero))
    seen = (r > 0).double()[:, None]
    grads = torch.autograd.grad([m2, conic, colors], [*leaves[:3], sh], [gm * seen, gc * seen, gcol])
    return [img[0], 0.5 * (diff ** 2).sum(), *grads[:3], go, grads[3]]
