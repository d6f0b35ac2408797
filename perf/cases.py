"""The measured cases of the renderer: what its users have it do, through the
public entry points of paper_2505_23158_gb300.api, over the range of sizes,
modes and directions that the library serves.

Scenes are the outdoor LOD scene of synth.workload_outdoor (16 level-0
Gaussians per square metre on a heightfield, four levels, chunk cells of
62.5 m, thresholds 10 / 20 / 40 m) at several extents, the plain 4,096-Gaussian
scene of config 0, and the dense chunk cell of the fine-tuning configuration.
Parameters are drawn on the GPU from the seed, so that a case is prepared in
about a second; cameras come from synth with the same seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2505_23158_gb300 import synth
from paper_2505_23158_gb300.api import (CHUNK, CHUNK_BLEND, FULL, LOD, Lodge, render_differentiable,
                                        render_level_lod)

MODES = {"FULL": FULL, "LOD": LOD, "CHUNK": CHUNK, "CHUNK_BLEND": CHUNK_BLEND}
DENSITY = 16.0          # level-0 Gaussians per square metre (16M on 1 km^2)
CELL = 62.5             # chunk cell, metres
THRESHOLDS = (10.0, 20.0, 40.0)
MIP_VARS = (0.0, 4e-4, 1.6e-3, 6.4e-3)   # Eq. 3 variance per level where the filters are on


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _render(name, mode, n0, w, h, cams, via="device", mip=False, sh=3):
    c = dict(kind="render", mode=mode, n0=n0, width=w, height=h, cams=cams, via=via, mip=mip, sh_degree=sh)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one 256 x 256 view of the 4,096-Gaussian scene,
        # all launches and latency (thumbnails, tests, toy scenes)
        dict(name="plain_256", kind="plain", n=4096, width=256, height=256),
        # one frame of an interactive viewer: LOD + chunks + opacity blending
        # at 1080p, waited for before the next pose is known
        _render("chunk_blend_1080p_single", "CHUNK_BLEND", 1_600_000, 1920, 1080, 1),
        # a stretch of a camera path in one call (the headline throughput)
        _render("chunk_blend_1080p_path", "CHUNK_BLEND", 4_000_000, 1920, 1080, 24),
        # the same path at full detail, the paper's first row: every level-0
        # Gaussian, millions of small splats
        _render("full_1080p_path", "FULL", 4_000_000, 1920, 1080, 4),
        # LOD selection per frame, no chunks (scenes without a chunk grid)
        _render("lod_1080p_single", "LOD", 4_000_000, 1920, 1080, 1),
        # the large scene's camera batch at 4K
        _render("chunk_blend_4k_batch", "CHUNK_BLEND", 1_600_000, 3840, 2160, 4),
        # the paper's Zip-NeRF image size, ragged in tiles, with both
        # Mip-Splatting filters on and degree-2 SH, no blending
        _render("chunk_mip_1392x793", "CHUNK", 640_000, 1392, 793, 6, mip=True, sh=2),
        # images wanted in host memory (page-locked), copies included
        _render("host_1080p_path", "CHUNK_BLEND", 1_600_000, 1920, 1080, 12, via="host"),
        # one step of the serving loop: requests of different scenes, modes
        # and resolutions composited together
        dict(name="serve_step_12", kind="step", n0=640_000, n=4096, frames=12, width=1280, height=720),
        # a fine-tuning step of one level: forward, L1 loss, gradients of all
        # parameters (2M Gaussians of one chunk cell, 720p)
        dict(name="finetune_2m_720p", kind="finetune", n=2_000_000, width=1280, height=720),
        # a step of the per-level build: two levels rendered with LOD
        # thresholds, gradients of the coarser one, an odd image size
        dict(name="build_step_803x451", kind="build", n=400_000, n1=150_000, width=803, height=451),
        # visibility filtering of one chunk: importance scores of its set over
        # views drawn inside it
        dict(name="importance_720p_views", kind="importance", n0=640_000, width=1280, height=720, cams=6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo, hi):
    """An image: width log-uniform in [lo, hi], odd as often as not, one of
    the usual shapes."""
    w = _log_int(rng, lo, hi)
    return w, max(48, int(w / rng.choice([16 / 9, 4 / 3, 1.755])))


def draw(rng):
    kind = rng.choice(["plain", "render", "render", "render", "render", "host", "step", "finetune", "build",
                       "importance"])
    if kind == "plain":
        w, h = _size(rng, 64, 1024)
        return dict(kind="plain", n=_log_int(rng, 500, 60_000), width=w, height=h)
    if kind in ("render", "host"):
        w, h = _size(rng, 160, 3840)
        mode = rng.choice(["CHUNK_BLEND", "CHUNK_BLEND", "CHUNK", "LOD", "FULL"])
        n0 = _log_int(rng, 20_000, 2_500_000)
        big = (w * h) / (1920 * 1080)
        top = 4 if mode == "FULL" else 16
        return _render(None, mode, n0, w, h, max(1, min(rng.randint(1, top), int(16 / max(big, 0.5)))),
                       via="host" if kind == "host" else "device", mip=rng.random() < 0.3,
                       sh=rng.choice([0, 1, 2, 3, 3, 3]))
    if kind == "step":
        w, h = _size(rng, 320, 1920)
        return dict(kind="step", n0=_log_int(rng, 50_000, 1_000_000), n=_log_int(rng, 1000, 30_000),
                    frames=rng.randint(2, 16), width=w, height=h)
    if kind == "finetune":
        w, h = _size(rng, 200, 1280)
        return dict(kind="finetune", n=_log_int(rng, 10_000, 1_800_000), width=w, height=h)
    if kind == "build":
        w, h = _size(rng, 200, 1000)
        n = _log_int(rng, 20_000, 600_000)
        return dict(kind="build", n=n, n1=max(1000, int(n * rng.uniform(0.2, 0.6))), width=w, height=h)
    w, h = _size(rng, 200, 1600)
    return dict(kind="importance", n0=_log_int(rng, 50_000, 1_000_000), width=w, height=h, cams=rng.randint(1, 6))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed, *stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1_000_003 + sum((k + 1) * 7919 ** (i + 1) for i, k in enumerate(stream))) % (1 << 62))
    return g


def _height(hp, x, y):
    h = torch.zeros_like(x)
    for a, f, th, ph in zip(hp["a"], hp["f"], hp["theta"], hp["phi"]):
        h += a * torch.sin(2 * math.pi * f * (x * math.cos(th) + y * math.sin(th)) / 1000.0 + ph)
    return h


def _zorder(x, y, side):
    def spread(v):
        v = (v | (v << 8)) & 0x00FF00FF
        v = (v | (v << 4)) & 0x0F0F0F0F
        v = (v | (v << 2)) & 0x33333333
        return (v | (v << 1)) & 0x55555555

    qx = (x / side * 65535.0).clamp(0, 65535).to(torch.int64)
    qy = (y / side * 65535.0).clamp(0, 65535).to(torch.int64)
    return torch.argsort(spread(qx) | (spread(qy) << 1), stable=True)


def _terrain_level(seed, stream, l, n, hp, x0, y0, side):
    """Raw parameters of n Gaussians of level l on the heightfield square
    (x0, y0, side): the distributions of synth.outdoor_scene, drawn on the
    GPU."""
    g = _gen(seed, 1, stream)
    z = lambda k: torch.randn(n, k, generator=g, device="cuda", dtype=torch.float32)
    means = torch.empty(n, 3, device="cuda", dtype=torch.float64)
    means[:, :2] = torch.rand(n, 2, generator=g, device="cuda", dtype=torch.float64) * side
    means[:, 0] += x0
    means[:, 1] += y0
    means[:, 2] = _height(hp, means[:, 0], means[:, 1])
    means = (means + z(3).double() * (0.5 * 2.0 ** l)).float()
    logs = z(3) * 0.5 + (math.log(0.125) + l * math.log(2.0))
    quats, logits, sh = z(4), z(1)[:, 0] + 1.0, z(48) * 0.2
    p = _zorder(means[:, 0] - x0, means[:, 1] - y0, side)
    return [t[p].contiguous() for t in (means, logs, quats, logits, sh)]


def _plain_level(seed, n):
    """The distributions of synth.plain_scene."""
    g = _gen(seed, 2)
    z = lambda k: torch.randn(n, k, generator=g, device="cuda", dtype=torch.float32)
    means = torch.rand(n, 3, generator=g, device="cuda", dtype=torch.float32) * 2 - 1
    return [means, z(3) * 0.5 - 3.5, z(4), z(1)[:, 0].contiguous(), z(48) * 0.2]


def _outdoor(seed, n0, mip=False, sh_degree=3):
    """(per-level GPU parameters, the scene as a user loads it)."""
    side = math.sqrt(n0 / DENSITY)
    grid = max(1, int(round(side / CELL)))
    hp = synth.height_params(seed)
    levels = [_terrain_level(seed, l, l, max(n0 // 4 ** l, 1), hp, 0.0, 0.0, side) for l in range(4)]
    cc = (np.arange(grid) + 0.5) * (side / grid)
    gx, gy = np.meshgrid(cc, cc, indexing="xy")
    centers = np.stack([gx.ravel(), gy.ravel(), synth.height(hp, gx.ravel(), gy.ravel()) + 2.0], axis=1)
    fv = MIP_VARS if mip else (0.0,) * 4
    scene = synth.Scene(levels=[_host_level(t, v) for t, v in zip(levels, fv)],
                        d_thresholds=np.asarray(THRESHOLDS), chunk_centers=centers, sh_degree=sh_degree,
                        extent=side, height_params=hp, filter2d=mip)
    return levels, scene


def _host_level(t, filter_var=0.0):
    a = [x.cpu().numpy() for x in t]
    return synth.Level(a[0], a[1], a[2], a[3], a[4].reshape(-1, 16, 3), filter_var)


def _path(scene, seed, n, w, h):
    """n consecutive poses of a 60-pose street-level path from a seeded
    start."""
    poses = synth.outdoor_trajectory(scene, seed=seed, n_poses=60, width=w, height_px=h)
    k = int(np.random.default_rng(seed).integers(0, 60 - n + 1))
    return poses[k:k + n]


def _cams(case, scene, seed):
    if case["width"] * case["height"] > 2_400_000:   # 4K: a batch of unrelated street cameras
        return synth.random_street_cameras(scene, seed + 5, case["cams"], case["width"], case["height"])
    return _path(scene, seed, case["cams"], case["width"], case["height"])


def _plain_cam(case):
    return synth.plain_camera(case["width"], case["height"])


def _cell(case, seed, n, stream=10):
    """One dense chunk cell of level-0 Gaussians (the fine-tuning
    configuration: the cell holds n) and a view around it looking inward."""
    hp = synth.height_params(seed)
    lv = _terrain_level(seed, stream, 0, n, hp, 500 - CELL / 2, 500 - CELL / 2, CELL)
    holder = synth.Scene(levels=[], d_thresholds=np.zeros(0), chunk_centers=np.zeros((1, 3)), extent=1000.0,
                         height_params=hp)
    return lv, synth.finetune_cameras(holder, seed=seed, n=1, width=case["width"], height_px=case["height"])[0]


def _target(case, seed):
    return torch.rand(case["height"], case["width"], 3, generator=_gen(seed, 4), device="cuda")


def _step_frames(case, scene, plain_cam, seed):
    """Requests of a serving step: mostly chunk frames at the step's
    resolution, some at other sizes and modes, a few of a small scene."""
    poses = synth.random_street_cameras(scene, seed + 5, case["frames"], case["width"], case["height"])
    small = synth.random_street_cameras(scene, seed + 6, case["frames"], max(case["width"] // 2 - 1, 64),
                                        max(case["height"] // 2 - 1, 48))
    out = []
    for i in range(case["frames"]):
        if i % 6 == 5:
            out.append((1, "FULL", plain_cam))
        elif i % 4 == 2:
            out.append((0, "LOD", small[i]))
        elif i % 4 == 3:
            out.append((0, "CHUNK", poses[i]))
        else:
            out.append((0, "CHUNK_BLEND", poses[i]))
    return out


def _image_buffer(case):
    return torch.empty(case["cams"] * case["width"] * case["height"] * 3, device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "ctx": Lodge(torch.cuda.current_device())}
    ctx = st["ctx"]
    if kind == "plain":
        lv = _plain_level(seed, case["n"])
        sc = synth.Scene(levels=[_host_level(lv)], d_thresholds=np.zeros(0), chunk_centers=np.zeros((1, 3)))
        st.update(sid=ctx.load_scene(sc), cam=_plain_cam(case),
                  out=torch.empty(case["width"] * case["height"] * 3, device="cuda"))
    elif kind == "render":
        _, scene = _outdoor(seed, case["n0"], case["mip"], case["sh_degree"])
        st.update(sid=ctx.load_scene(scene), cams=_cams(case, scene, seed))
        if case["via"] == "host":
            px = case["width"] * case["height"] * 3
            st["host"] = torch.empty(case["cams"] * px, pin_memory=True).numpy()
        else:
            st["out"] = _image_buffer(case)
    elif kind == "step":
        _, scene = _outdoor(seed, case["n0"])
        lv = _plain_level(seed, case["n"])
        sc = synth.Scene(levels=[_host_level(lv)], d_thresholds=np.zeros(0), chunk_centers=np.zeros((1, 3)))
        sids = [ctx.load_scene(scene), ctx.load_scene(sc)]
        pc = synth.plain_camera(case["width"] // 2, case["height"] // 2)
        st["frames"] = [(sids[s], MODES[m], c) for s, m, c in _step_frames(case, scene, pc, seed)]
    elif kind == "finetune":
        lv, cam = _cell(case, seed, case["n"])
        st.update(params=[t.requires_grad_(True) for t in lv], cam=cam, target=_target(case, seed))
    elif kind == "build":
        fixed, trained, cam, d, fv = _build_inputs(case, seed)
        st.update(fixed=fixed, params=[t.requires_grad_(True) for t in trained], cam=cam, d=d, fv=fv,
                  target=_target(case, seed))
    elif kind == "importance":
        _, scene = _outdoor(seed, case["n0"])
        chunk = _chunk_of(scene, seed)
        st.update(sid=ctx.load_scene(scene), chunk=chunk, n=scene.n_total,
                  cams=synth.chunk_views(scene, chunk, seed, case["cams"], case["width"], case["height"]))
    return st


def _chunk_of(scene, seed):
    return int(np.random.default_rng(seed).integers(0, scene.chunk_centers.shape[0]))


def _build_inputs(case, seed):
    fixed, cam = _cell(case, seed, case["n"])
    trained, _ = _cell(case, seed, case["n1"], 11)
    d = float(np.random.default_rng(seed).uniform(0.7, 1.3)) * THRESHOLDS[0]
    return [tuple(fixed)], trained, cam, [d], [0.0, 4e-4]


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
COUNTS = ("n_active", "n_visible", "n_keys", "n_tiles")


def _counts(stats):
    return np.asarray([[s[k] for k in COUNTS] for s in stats], np.int64)


def run(st):
    case, ctx = st["case"], st["ctx"]
    kind = case["kind"]
    if kind == "plain":
        img, stats = ctx.render(st["sid"], FULL, st["cam"], out=st["out"])
        return {"images": [img], "counts": _counts([stats])}
    if kind == "render":
        mode = MODES[case["mode"]]
        if case["via"] == "host":
            stats = ctx.render_host(st["sid"], mode, st["cams"], st["host"])
            return {"images": list(st["host"].reshape(case["cams"], case["height"], case["width"], 3)),
                    "counts": _counts(stats)}
        if case["cams"] == 1:
            img, s = ctx.render(st["sid"], mode, st["cams"][0], out=st["out"])
            return {"images": [img], "counts": _counts([s])}
        imgs, stats = ctx.render(st["sid"], mode, st["cams"], out=st["out"])
        return {"images": imgs, "counts": _counts(stats)}
    if kind == "step":
        imgs, stats = ctx.render_batch(st["frames"])
        return {"images": imgs, "counts": _counts(stats)}
    if kind == "finetune":
        img = render_differentiable(ctx, *st["params"], st["cam"])
        loss = (img - st["target"]).abs().mean()
        return {"images": [img.detach()], "grads": list(torch.autograd.grad(loss, st["params"]))}
    if kind == "build":
        img = render_level_lod(ctx, st["params"], st["fixed"], 1, st["cam"], st["d"], st["fv"])
        loss = (img - st["target"]).abs().mean()
        return {"images": [img.detach()], "grads": list(torch.autograd.grad(loss, st["params"]))}
    return {"score": ctx.importance(st["sid"], CHUNK, st["cams"], chunk=st["chunk"])}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _loaded(mode, n0):
    """Gaussians a frame loads: all of level 0, or the Eq. 2 rings (per metre
    of radius) with the chunk radius added to the thresholds."""
    if mode == "FULL":
        return n0
    area = n0 / DENSITY
    r = CELL if mode != "LOD" and area > 2 * CELL * CELL else 0.0
    edges = [0.0] + [d + r for d in THRESHOLDS] + [1e9]
    total = 0.0
    for l in range(4):
        inner = min(math.pi * edges[l] ** 2, area)
        outer = min(math.pi * edges[l + 1] ** 2, area)
        total += (outer - inner) * DENSITY / 4 ** l
    return total * (1.5 if mode == "CHUNK_BLEND" and r else 1.0)


def _frame_work(loaded, pixels, visible=0.25, per_pixel=30):
    """A frame reads the mean of every loaded Gaussian and the other 224 B of
    the visible ones, and writes 12 B a pixel; about 500 operations project a
    visible Gaussian, about 15 composite one at a pixel."""
    return (loaded * (12 + 224 * visible) + 12 * pixels, 500 * loaded * visible + 15 * per_pixel * pixels)


def work(case):
    kind, px = case["kind"], case["width"] * case["height"]
    if kind == "plain":
        b, f = _frame_work(case["n"], px, 1.0, 20)
    elif kind == "render":
        b, f = (case["cams"] * x for x in _frame_work(_loaded(case["mode"], case["n0"]), px))
    elif kind == "step":
        b, f = (case["frames"] * x for x in _frame_work(_loaded("CHUNK_BLEND", case["n0"]), 0.75 * px))
    elif kind == "importance":
        b, f = (case["cams"] * x for x in _frame_work(_loaded("CHUNK", case["n0"]), px))
    else:
        # parameters read by both directions, gradients written; the adjoint
        # takes about three times the forward's operations at a pixel
        n = case["n"] + case.get("n1", 0)
        trained = case.get("n1", case["n"])
        b = 236 * n + 2 * 236 * trained + 2 * 12 * px
        f = 2000 * n * 0.3 + 60 * 40 * px
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# the same in 64 bits, plain torch
# ---------------------------------------------------------------------------
def _sh_basis(d):
    x, y, z = d.unbind(-1)
    xx, yy, zz = x * x, y * y, z * z
    s = math.sqrt
    pi = math.pi
    return torch.stack([
        torch.full_like(x, 0.5 / s(pi)),
        s(3 / (4 * pi)) * y, s(3 / (4 * pi)) * z, s(3 / (4 * pi)) * x,
        0.5 * s(15 / pi) * x * y, 0.5 * s(15 / pi) * y * z, 0.25 * s(5 / pi) * (3 * zz - 1),
        0.5 * s(15 / pi) * x * z, 0.25 * s(15 / pi) * (xx - yy),
        0.25 * s(35 / (2 * pi)) * y * (3 * xx - yy), 0.5 * s(105 / pi) * x * y * z,
        0.25 * s(21 / (2 * pi)) * y * (5 * zz - 1), 0.25 * s(7 / pi) * z * (5 * zz - 3),
        0.25 * s(21 / (2 * pi)) * x * (5 * zz - 1), 0.25 * s(105 / pi) * z * (xx - yy),
        0.25 * s(35 / (2 * pi)) * x * (xx - 3 * yy)], -1)


def _project64(p, cam, var, mult, filter2d, sh_degree):
    """Raw parameters (64 bits) to the 2D quantities of the near-culled ones:
    dict of mean, conic, opacity, colour, depth, covariance diagonal, and the
    kept indices."""
    dev = p[0].device
    R = torch.as_tensor(np.asarray(cam.R, np.float64), device=dev)
    t = torch.as_tensor(np.asarray(cam.t, np.float64), device=dev)
    c = torch.as_tensor(np.asarray(cam.center, np.float64), device=dev)
    keep = ((p[0] @ R.T + t)[:, 2] > float(np.float32(cam.znear))).nonzero()[:, 0]
    means, logs, quats, logits, sh = [x[keep] for x in p]
    var, mult = var[keep], mult[keep]
    pc = means @ R.T + t
    x, y, z = pc.unbind(-1)
    fx, fy, cx, cy = (float(np.float32(v)) for v in (cam.fx, cam.fy, cam.cx, cam.cy))
    s = torch.exp(logs)
    sig = torch.sqrt(s * s + var[:, None])
    op = torch.sigmoid(logits) * mult * (s / sig).prod(-1)
    q = quats / quats.norm(dim=-1, keepdim=True)
    w, qx, qy, qz = q.unbind(-1)
    M = torch.stack([1 - 2 * (qy * qy + qz * qz), 2 * (qx * qy - w * qz), 2 * (qx * qz + w * qy),
                     2 * (qx * qy + w * qz), 1 - 2 * (qx * qx + qz * qz), 2 * (qy * qz - w * qx),
                     2 * (qx * qz - w * qy), 2 * (qy * qz + w * qx), 1 - 2 * (qx * qx + qy * qy)],
                    -1).view(-1, 3, 3)
    limx, limy = 1.3 * cam.width / (2 * fx), 1.3 * cam.height / (2 * fy)
    uc, wc = (x / z).clamp(-limx, limx), (y / z).clamp(-limy, limy)
    o = torch.zeros_like(z)
    J = torch.stack([torch.stack([fx / z, o, -fx * uc / z], -1), torch.stack([o, fy / z, -fy * wc / z], -1)], -2)
    B = (J @ R) @ M * sig[:, None, :]
    S = B @ B.transpose(1, 2)
    a, b, cc = S[:, 0, 0] + 0.3, S[:, 0, 1], S[:, 1, 1] + 0.3
    det = a * cc - b * b
    if filter2d:
        det0 = S[:, 0, 0] * S[:, 1, 1] - S[:, 0, 1] ** 2
        op = op * torch.sqrt((det0 / det).clamp(min=0))
    d = means - c
    d = d / d.norm(dim=-1, keepdim=True)
    nk = (sh_degree + 1) ** 2
    rgb = ((_sh_basis(d)[:, :nk, None] * sh.view(-1, 16, 3)[:, :nk]).sum(1) + 0.5).clamp(min=0)
    return dict(mean=torch.stack([fx * x / z + cx, fy * y / z + cy], -1),
                conic=torch.stack([cc / det, -b / det, a / det], -1), op=op, rgb=rgb,
                z=z.detach(), a=a.detach(), c=cc.detach(), keep=keep)


BLOCK = 32   # pixels per side of the blocks composited at once


def _composite64(v, cam, grad_image=None, want_score=False):
    """Image of the projected quantities, block by block: per block the
    Gaussians that can reach alpha >= 1/255 in it, in depth order.  With
    grad_image(image block, rows, columns) -> dL/dblock also the gradients of
    mean, conic, op and rgb; with want_score each Gaussian's largest weight."""
    H, W = cam.height, cam.width
    dev = v["z"].device
    with torch.no_grad():
        order = torch.argsort(v["z"].float(), stable=True)   # the depth key is the rounded depth
        order = order[v["op"][order] >= (1 / 255) * (1 - 1e-6)]
        mean, op = v["mean"][order], v["op"][order]
        Q = 2 * torch.log((255 * op).clamp(min=1)) + 0.05
        rx, ry = torch.sqrt(Q * v["a"][order]) + 1, torch.sqrt(Q * v["c"][order]) + 1
        x0, x1, y0, y1 = mean[:, 0] - rx, mean[:, 0] + rx, mean[:, 1] - ry, mean[:, 1] + ry
        on = (x1 > 0) & (x0 < W) & (y1 > 0) & (y0 < H)
        order, x0, x1, y0, y1 = order[on], x0[on], x1[on], y0[on], y1[on]
    img = torch.zeros(H, W, 3, dtype=torch.float64, device=dev)
    names = ("mean", "conic", "op", "rgb")
    src = {k: v[k].detach() for k in names}
    grads = {k: torch.zeros_like(src[k]) for k in names} if grad_image else None
    score = torch.zeros(v["z"].numel(), dtype=torch.float64, device=dev) if want_score else None
    for by in range(0, H, BLOCK):
        rows = ((y1 > by) & (y0 < by + BLOCK)).nonzero()[:, 0]
        o_r, x0_r, x1_r = order[rows], x0[rows], x1[rows]
        for bx in range(0, W, BLOCK):
            idx = o_r[(x1_r > bx) & (x0_r < bx + BLOCK)]
            if not idx.numel():
                continue
            py = torch.arange(by, min(by + BLOCK, H), device=dev, dtype=torch.float64) + 0.5
            px = torch.arange(bx, min(bx + BLOCK, W), device=dev, dtype=torch.float64) + 0.5
            t = {k: src[k][idx].requires_grad_(grads is not None) for k in names}
            with torch.enable_grad() if grads is not None else torch.no_grad():
                dx = px[None, :, None] - t["mean"][:, 0]
                dy = py[:, None, None] - t["mean"][:, 1]
                cn = t["conic"]
                e = -0.5 * (cn[:, 0] * dx * dx + cn[:, 2] * dy * dy) - cn[:, 1] * dx * dy
                alpha = (t["op"] * torch.exp(e)).clamp(max=0.99)
                alpha = torch.where(alpha >= 1 / 255, alpha, torch.zeros_like(alpha))
                after = torch.cumsum(torch.log1p(-alpha), -1)
                with torch.no_grad():
                    live = after >= math.log(1e-4)
                T = torch.exp(after - torch.log1p(-alpha))
                wgt = torch.where(live, T * alpha, torch.zeros_like(alpha))
                block = wgt @ t["rgb"]
            img[by:by + BLOCK, bx:bx + BLOCK] = block.detach()
            if grads is not None:
                g = grad_image(block.detach(), slice(by, by + py.numel()), slice(bx, bx + px.numel()))
                for k, gk in zip(names, torch.autograd.grad(block, [t[k] for k in names], g)):
                    grads[k].index_add_(0, idx, gk)
            if score is not None:
                best = wgt.detach().reshape(-1, idx.numel()).amax(0)
                score[idx] = torch.maximum(score[idx], best)
    return img, grads, score


def _bands(d):
    """Squared Eq. 2 bands as the selection takes them: FP32."""
    e = [0.0] + [float(np.float32(x * x)) for x in d] + [math.inf]
    return list(zip(e[:-1], e[1:]))


def _select(levels, center, d):
    """Per level, whether Eq. 2 holds: squared FP32 distances."""
    c = torch.as_tensor(np.asarray(center, np.float64).astype(np.float32), device="cuda")
    out = []
    for lv, (lo, hi) in zip(levels, _bands(d)):
        q = (lv[0] - c).square()
        D = (q[:, 0] + q[:, 1]) + q[:, 2]
        out.append((D >= lo) & (D < hi))
    return torch.cat(out)


def _radius(centers, k):
    if len(centers) < 2:
        return 0.0
    d = np.linalg.norm(centers - centers[k], axis=1)
    return float(np.delete(d, k).min())


def _active(levels, centers, mode, cam):
    """(mask over all levels, opacity multiplier)."""
    n = [lv[0].shape[0] for lv in levels]
    one = torch.ones(sum(n), dtype=torch.float64, device="cuda")
    if mode == "FULL":
        m = torch.zeros(sum(n), dtype=torch.bool, device="cuda")
        m[:n[0]] = True
        return m, one
    if mode == "LOD":
        return _select(levels, cam.center, THRESHOLDS), one
    d2 = ((centers - cam.center) ** 2).sum(1)
    order = np.argsort(d2, kind="stable")
    A = int(order[0])
    of = lambda k: _select(levels, centers[k], [t + _radius(centers, k) for t in THRESHOLDS])
    mA = of(A)
    if mode == "CHUNK" or len(order) < 2:
        return mA, one
    B = int(order[1])
    mB = of(B)
    ab = centers[A] - centers[B]
    tA = float(np.clip((cam.center - centers[B]) @ ab / (ab @ ab), 0, 1))
    tB = float(np.clip((cam.center - centers[A]) @ -ab / (ab @ ab), 0, 1))
    mult = one.clone()
    mult[mA & ~mB] = tA
    mult[mB & ~mA] = tB
    return mA | mB, mult


def _frame64(levels, mask, mult, cam, fv, filter2d, sh_degree, **kw):
    sel = mask.nonzero()[:, 0]
    p = [torch.cat([lv[k] for lv in levels])[sel].double() for k in range(5)]
    var = torch.cat([torch.full((lv[0].shape[0],), float(np.float32(f)), dtype=torch.float64, device="cuda")
                     for lv, f in zip(levels, fv)])[sel]
    v = _project64(p, cam, var, mult[sel], filter2d, sh_degree)
    return sel, v, _composite64(v, cam, **kw)


def _exact_grads(levels, mask, cam, fv, target, trained):
    """Image and the gradients of the mean absolute difference to target with
    respect to the trained level's parameters."""
    sel = mask.nonzero()[:, 0]
    n = [lv[0].shape[0] for lv in levels]
    p = [torch.cat([lv[k].detach() for lv in levels])[sel].double().requires_grad_(True) for k in range(5)]
    var = torch.cat([torch.full((m,), float(np.float32(f)), dtype=torch.float64, device="cuda")
                     for m, f in zip(n, fv)])[sel]
    v = _project64(p, cam, var, torch.ones_like(var), False, 3)
    tgt = target.double()
    img, g, _ = _composite64(v, cam, grad_image=lambda b, r, c: torch.sign(b - tgt[r, c]) / tgt.numel())
    names = ("mean", "conic", "op", "rgb")
    gp = torch.autograd.grad([v[k] for k in names], p, [g[k] for k in names])
    lo = sum(n[:trained])
    full = []
    for k, x in enumerate(gp):
        out = torch.zeros((sum(n),) + tuple(x.shape[1:]), dtype=torch.float64, device="cuda")
        out[sel] = x
        full.append(out[lo:lo + n[trained]])
    return {"images": [img], "grads": full}


def exact(case, seed):
    kind = case["kind"]
    if kind == "plain":
        lv = [_plain_level(seed, case["n"])]
        m = torch.ones(case["n"], dtype=torch.bool, device="cuda")
        _, _, (img, _, _) = _frame64(lv, m, m.double(), _plain_cam(case), [0.0], False, 3)
        return {"images": [img], "counts": None}
    if kind == "render":
        levels, scene = _outdoor(seed, case["n0"], case["mip"], case["sh_degree"])
        cams = _cams(case, scene, seed)
        imgs = []
        for i, cam in enumerate(cams):
            if i:   # one frame of a path: the others are alike
                imgs.append(None)
                continue
            m, mult = _active(levels, scene.chunk_centers, case["mode"], cam)
            fv = MIP_VARS if case["mip"] else (0.0,) * 4
            _, _, (img, _, _) = _frame64(levels, m, mult, cam, fv, case["mip"], case["sh_degree"])
            imgs.append(img)
        return {"images": imgs, "counts": None}
    if kind == "step":
        levels, scene = _outdoor(seed, case["n0"])
        pc = synth.plain_camera(case["width"] // 2, case["height"] // 2)
        imgs = []
        for i, (s, mode, cam) in enumerate(_step_frames(case, scene, pc, seed)):
            if i > 3:
                imgs.append(None)
                continue
            lv = levels if s == 0 else [_plain_level(seed, case["n"])]
            m, mult = _active(lv, scene.chunk_centers, mode, cam)
            _, _, (img, _, _) = _frame64(lv, m, mult, cam, (0.0,) * 4, False, 3)
            imgs.append(img)
        return {"images": imgs, "counts": None}
    if kind == "finetune":
        lv, cam = _cell(case, seed, case["n"])
        m = torch.ones(case["n"], dtype=torch.bool, device="cuda")
        return _exact_grads([lv], m, cam, [0.0], _target(case, seed), 0)
    if kind == "build":
        fixed, trained, cam, d, fv = _build_inputs(case, seed)
        levels = fixed + [tuple(trained)]
        return _exact_grads(levels, _select(levels, cam.center, d), cam, fv, _target(case, seed), 1)
    levels, scene = _outdoor(seed, case["n0"])
    k = _chunk_of(scene, seed)
    m = _select(levels, scene.chunk_centers[k], [t + _radius(scene.chunk_centers, k) for t in THRESHOLDS])
    score = torch.zeros(scene.n_total, dtype=torch.float64, device="cuda")
    for cam in synth.chunk_views(scene, k, seed, case["cams"], case["width"], case["height"]):
        sel, v, (_, _, s) = _frame64(levels, m, m.double(), cam, (0.0,) * 4, False, 3, want_score=True)
        at = sel[v["keep"]]
        score[at] = torch.maximum(score[at], s)
    return {"score": score}
