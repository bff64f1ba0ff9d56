"""Performance cases of the rasteriser: what its users have it do, through its
public entry points.

listed() names the cases, draw() draws more of the same ranges, prepare()
makes what a caller holds before the call (scene, cameras, the kept frame or
batch), run() makes one pass, work() states what a pass cannot do without, and
exact() computes the outputs in float64 with plain torch.

Kinds of pass:
  call    rasterizer.forward on a kept frame (one view, the pair count read back)
  frame   a kept frame's stages preprocess, bin_emit, sort, render (a render loop)
  grad    rasterizer.rasterize and its backward (autograd)
  back    qb_render_bwd alone on a rendered frame
  train   rasterizer.Trainer.step
  batch   rasterizer.Batch.render over many cameras
  bgrad   Batch.render and Batch.backward
  sort    qb_sort_pairs alone
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2605_04844_gb300 import _native as N
from paper_2605_04844_gb300 import rasterizer as R

KEYS = ("means", "scales", "quats", "opacities", "sh")
RESOLUTIONS = ((800, 800), (1264, 832), (1600, 900), (1920, 1080))
ZNEAR = 0.2
FOV_X = 60.0


def listed():
    return [
        # a thumbnail or an interactive preview: 10k Gaussians without SH bands, where
        # launches and the host's part of a call count
        dict(name="call_10k_256", kind="call", scene="uniform", n=10_000, w=256, h=256, deg=0, mode="quadbox"),
        # a step of a small fit with the user's own loss, through autograd; ragged image
        dict(name="grad_20k_ragged", kind="grad", scene="uniform", n=20_011, w=333, h=217, deg=1, mode="quadbox"),
        # a render loop over a middle-sized scene with second-degree SH, ragged image
        dict(name="frame_200k_ragged", kind="frame", scene="blobs", n=200_003, w=1001, h=701, deg=2, mode="quadbox"),
        # the headline frame: 1M Gaussians, 1080p, SH degree 3
        dict(name="frame_1m_1080p", kind="frame", scene="blobs", n=1_000_000, w=1920, h=1080, deg=3, mode="quadbox"),
        # the same frame with the 3-sigma box of 3DGS, which users compare with (three times the pairs)
        dict(name="frame_1m_1080p_aabb", kind="frame", scene="blobs", n=1_000_000, w=1920, h=1080, deg=3,
             mode="aabb3s"),
        # a large scene seen from inside at 1440p (the near half of the zoom sweep)
        dict(name="frame_3m_1440p_near", kind="frame", scene="ball", n=3_000_000, w=2560, h=1440, deg=3,
             mode="quadbox", dist=4.0),
        # a 4K frame (32400 tiles)
        dict(name="frame_1m_4k", kind="frame", scene="blobs", n=1_000_000, w=3840, h=2160, deg=3, mode="quadbox"),
        # the backward alone at the headline size, as a caller that computes its loss itself runs it
        dict(name="back_1m_1080p", kind="back", scene="blobs", n=1_000_000, w=1920, h=1080, deg=3, mode="quadbox"),
        # a training step: forward, L1 loss, backward and Adam on 500k Gaussians
        dict(name="train_500k", kind="train", scene="blobs", n=500_000, w=1264, h=832, deg=3, mode="quadbox"),
        # a light field or an evaluation set: sixteen views of one scene at mixed resolutions
        dict(name="batch_16x1m", kind="batch", scene="ball", n=1_000_000, cams=16, w=1920, h=1080, deg=3,
             mode="quadbox", dist=8.0),
        # a multi-view training step: gradients summed over a few views
        dict(name="bgrad_5x200k", kind="bgrad", scene="ball", n=200_004, cams=5, w=1264, h=832, deg=3,
             mode="quadbox", dist=8.0),
        # the pair sort alone, at the key width of a 1080p frame
        dict(name="sort_5m_44b", kind="sort", n=5_000_003, bits=44, digit=8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("call", "frame", "frame", "frame", "grad", "back", "train", "batch", "bgrad", "sort"))
    if kind == "sort":
        return dict(kind="sort", n=_log(rng, 10_000, 20_000_000), bits=rng.choice((39, 42, 44, 45, 46, 64)),
                    digit=rng.choice((8, 8, 11)))
    c = dict(kind=kind, deg=rng.choice((0, 1, 2, 3, 3)), mode="quadbox")
    if kind == "call":
        c.update(scene="uniform", n=_log(rng, 2_000, 100_000), w=_log(rng, 64, 1000), h=_log(rng, 64, 800))
    elif kind == "frame":
        c.update(scene=rng.choice(("blobs", "ball")), n=_log(rng, 20_000, 3_000_000), w=_log(rng, 300, 3840),
                 h=_log(rng, 300, 2160))
        if c["scene"] == "ball":
            c["dist"] = round(math.exp(rng.uniform(math.log(3.0), math.log(40.0))), 2)
        elif c["n"] <= 1_000_000 and c["w"] * c["h"] <= 2_100_000:
            c["mode"] = rng.choice(("quadbox", "quadbox", "adr", "aabb3s"))
    elif kind in ("grad", "back", "train"):
        c.update(scene=rng.choice(("uniform", "blobs")), n=_log(rng, 5_000, 1_000_000), w=_log(rng, 100, 1920),
                 h=_log(rng, 100, 1080))
        if c["scene"] == "uniform":
            c["n"] = min(c["n"], 100_000)
    else:
        cams = rng.randint(2, 16 if kind == "batch" else 8)
        # (a multiple of 4: the batch reads a camera's depth order 16 bytes at a time)
        c.update(scene="ball", n=4 * _log(rng, 5_000, 250_000 if kind == "batch" else 100_000), cams=cams,
                 w=1920, h=1080, dist=8.0)
    return c


# ---- inputs ------------------------------------------------------------------------------------


def _look_at(campos):
    """World->view matrix of a camera at campos looking at the origin (+y up)."""
    c = np.asarray(campos, dtype=np.float64)
    z = -c / np.linalg.norm(c)
    x = np.cross([0.0, 1.0, 0.0], z)
    x /= np.linalg.norm(x)
    V = np.eye(4)
    V[0, :3], V[1, :3], V[2, :3] = x, np.cross(z, x), z
    V[:3, 3] = -V[:3, :3] @ c
    return V


def _camera(w, h, V=None):
    tanx = math.tan(math.radians(FOV_X) / 2.0)
    f = w / (2.0 * tanx)
    V = np.eye(4) if V is None else V
    return {"viewmat": V.astype(np.float32), "fx": f, "fy": f, "cx": (w - 1) / 2.0, "cy": (h - 1) / 2.0,
            "tan_fovx": tanx, "tan_fovy": h / (2.0 * f), "campos": (-V[:3, :3].T @ V[:3, 3]).astype(np.float32),
            "width": w, "height": h, "znear": ZNEAR}


def _cameras(case, seed):
    w, h = case["w"], case["h"]
    if case["scene"] != "ball":
        return [_camera(w, h)]
    if "cams" not in case:
        return [_camera(w, h, _look_at((0.0, 0.0, -case["dist"])))]
    # a Fibonacci lattice on a sphere around the scene, turned by the seed
    rng = np.random.default_rng(seed)
    turn = rng.uniform(0.0, 2.0 * math.pi)
    cams = []
    for k in range(case["cams"]):
        y = 1.0 - 2.0 * (k + 0.5) / case["cams"]
        r, th = math.sqrt(1.0 - y * y), turn + math.pi * (3.0 - math.sqrt(5.0)) * k
        pos = case["dist"] * np.array([r * math.cos(th), y, r * math.sin(th)])
        w, h = RESOLUTIONS[k % len(RESOLUTIONS)]
        cams.append(_camera(w, h, _look_at(pos)))
    return cams


def _scene(case, seed, dev):
    """Raw parameters: clustered scenes (64 blobs and a fifth of the Gaussians
    as background, a tenth of them long), or one uniform in the frustum."""
    g = torch.Generator(dev).manual_seed(int(seed))
    n, deg, kind = case["n"], case["deg"], case["scene"]

    def uni(*shape):
        return torch.rand(shape, generator=g, device=dev)

    def nrm(*shape):
        return torch.randn(shape, generator=g, device=dev)

    tanx = math.tan(math.radians(FOV_X) / 2.0)
    tany = tanx * case["h"] / case["w"]

    def frustum(m, lo, hi):
        z = lo + (hi - lo) * uni(m)
        return torch.stack([(2 * uni(m) - 1) * z * tanx, (2 * uni(m) - 1) * z * tany, z], 1)

    def ball(m, radius):
        d = nrm(m, 3)
        return d / d.norm(dim=1, keepdim=True) * (radius * uni(m, 1) ** (1.0 / 3.0))

    if kind == "uniform":
        means = frustum(n, 2.0, 6.0)
        scales = -3.5 + 0.8 * nrm(n, 3)
        logits = 1.5 * nrm(n)
    else:
        nb = int(round(0.8 * n))
        radius = 4.0 if "cams" in case else 10.0
        centre = frustum(64, 1.0, 50.0) if kind == "blobs" else ball(64, radius)
        which = torch.randint(0, 64, (nb,), generator=g, device=dev)
        c = centre[which]
        blob = c + nrm(nb, 3) * (0.05 * c[:, 2:3] if kind == "blobs" else 0.5)
        rest = frustum(n - nb, 1.0, 50.0) if kind == "blobs" else ball(n - nb, radius)
        means = torch.cat([blob, rest])[torch.randperm(n, generator=g, device=dev)]
        scales = -4.0 + nrm(n, 3)
        long = torch.nn.functional.one_hot(torch.randint(0, 3, (n,), generator=g, device=dev), 3)
        scales = scales + 2.5 * long * (uni(n, 1) < 0.1)
        logits = 2.0 * nrm(n)
    K = (deg + 1) ** 2
    sh = 0.1 * nrm(n, K, 3)
    sh[:, 0] = (uni(n, 3) - 0.5) * (2.0 * math.sqrt(math.pi))
    return {"means": means.contiguous(), "scales": scales.contiguous(), "quats": nrm(n, 4), "opacities": logits,
            "sh": sh.contiguous(), "sh_degree": deg, "raw": 1}


def _image_like(case, seed, what, shape, dev):
    """Per-pixel inputs of the backward: a target image, or a loss gradient."""
    g = torch.Generator(dev).manual_seed(int(seed) + 77_000)
    if what == "target":
        return torch.rand(shape, generator=g, device=dev)
    return torch.randn(shape, generator=g, device=dev) / math.prod(shape)


BG = (0.1, 0.2, 0.3)
LR = {"means": 1.6e-4, "scales": 5e-3, "quats": 1e-3, "opacities": 5e-2, "sh": 2.5e-3}
BETAS, EPS, RESUMED_AT = (0.9, 0.999), 1e-15, 1000


def _moments(scene, seed, dev):
    """Adam's moments of a training run resumed from a checkpoint."""
    g = torch.Generator(dev).manual_seed(int(seed) + 99_000)
    m, v = {}, {}
    for k in KEYS:
        m[k] = 1e-7 * torch.randn(scene[k].shape, generator=g, device=dev)
        v[k] = 1e-13 * (0.5 + torch.rand(scene[k].shape, generator=g, device=dev))
    return m, v


def _sort_input(case, seed, dev):
    g = torch.Generator(dev).manual_seed(int(seed))
    keys = torch.randint(-(2 ** 63), 2 ** 63 - 1, (case["n"],), generator=g, device=dev, dtype=torch.int64)
    if case["bits"] < 64:
        keys &= (1 << case["bits"]) - 1
    return keys, torch.arange(case["n"], dtype=torch.int32, device=dev)


def _grads_struct(grads):
    gs = N.QbSceneGrads()
    for k in KEYS:
        setattr(gs, k, grads[k].data_ptr())
    return gs


def prepare(case, seed):
    dev = "cuda"
    kind = case["kind"]
    if kind == "sort":
        keys, vals = _sort_input(case, seed, dev)
        need = N.qb_sort_scratch_bytes(case["n"], case["bits"], case["digit"])
        raw = torch.empty(need + 256, dtype=torch.uint8, device=dev)
        off = (-raw.data_ptr()) % 256
        return dict(case=case, keys=keys, vals=vals, scratch=raw[off:off + need],
                    work=[torch.empty_like(t) for t in (keys, vals, keys, vals)])
    scene, cams = _scene(case, seed, dev), _cameras(case, seed)
    st = dict(case=case, scene=scene, cams=cams, scene_s=R.scene_struct(scene))
    if kind in ("batch", "bgrad"):
        st["arr"] = R.camera_array(cams)
        st["batch"] = R.calibrated_batch(scene, cams, case["mode"])
        if kind == "bgrad":
            b = st["batch"]
            st["dL"] = _image_like(case, seed, "loss", tuple(b.images.shape), dev)
            st["grads"] = {k: torch.zeros_like(scene[k]) for k in KEYS}
        return st
    cam = cams[0]
    shape = (3, cam["height"], cam["width"])
    st["cam_s"] = R.camera_struct(cam)
    if kind == "grad":
        st["leaves"] = {k: scene[k].requires_grad_(True) for k in KEYS}
        st["dL"] = _image_like(case, seed, "loss", shape, dev)
    elif kind == "train":
        st["target"] = _image_like(case, seed, "target", shape, dev)
        tr = R.Trainer(scene, cam, case["mode"], lr=LR, betas=BETAS, eps=EPS, bg=BG)
        tr.m, tr.v = _moments(scene, seed, dev)
        tr.t = RESUMED_AT
        st["trainer"] = tr
    else:
        _, fr = R.forward(scene, cam, case["mode"], bg=BG)
        # the frame a render loop keeps: room for a tenth more pairs than this view has
        st["frame"] = R.Frame(case["n"], cam["width"], cam["height"], min(2 ** 30, int(fr.n_pairs * 1.1) + 4096))
        del fr
        if kind == "back":
            R.forward(scene, cam, case["mode"], bg=BG, frame=st["frame"])
            st["dL"] = _image_like(case, seed, "loss", shape, dev)
            st["grads"] = {k: torch.zeros_like(scene[k]) for k in KEYS}
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "sort":
        k, v, ka, va = st["work"]
        k.copy_(st["keys"])  # the sort is in place
        v.copy_(st["vals"])
        alt = N.qb_sort_pairs(k, v, ka, va, case["n"], case["bits"], case["digit"], st["scratch"])
        return [ka, va] if alt else [k, v]
    if kind == "call":
        img, st["frame"] = R.forward(st["scene"], st["cams"][0], case["mode"], bg=BG, frame=st["frame"])
        return img
    if kind == "frame":
        fr = st["frame"]
        fr.preprocess(st["scene_s"], st["cam_s"], case["mode"])
        fr.bin_emit(sync=False)
        fr.sort()
        return fr.render(BG)
    if kind == "grad":
        p = st["leaves"]
        img = R.rasterize(p["means"], p["scales"], p["quats"], p["opacities"], p["sh"], st["cams"][0], case["mode"],
                          BG)
        g = torch.autograd.grad(img, [p[k] for k in KEYS], st["dL"])
        return [img.detach(), *g]
    if kind == "back":
        for k in KEYS:
            st["grads"][k].zero_()  # the backward adds to them
        N.qb_render_bwd(st["frame"].frame, st["scene_s"], st["cam_s"], BG, st["dL"], _grads_struct(st["grads"]))
        return [st["grads"][k] for k in KEYS]
    if kind == "train":
        tr = st["trainer"]
        loss = tr.step(st["target"])
        return [loss.float(), tr.img, *[tr.grads[k] for k in KEYS], *[tr.scene[k] for k in KEYS]]
    b = st["batch"]
    images = b.render(st["scene_s"], st["arr"], case["mode"], bg=BG)
    if kind == "batch":
        return images
    for k in KEYS:
        st["grads"][k].zero_()
    b.backward(st["scene_s"], st["arr"], st["dL"], _grads_struct(st["grads"]), bg=BG)
    return [images, *[st["grads"][k] for k in KEYS]]


def work(case):
    """Bytes: every input read once and every output written once.  Operations:
    the projection of each Gaussian (about 400) and, per pixel, the entries it
    composites before it stops (about 70 in these scenes, 21 each; three times
    that in the backward)."""
    n = case["n"]
    if case["kind"] == "sort":
        return {"bytes": 24.0 * n, "flops": 0.0}
    params = 4.0 * n * (11 + 3 * (case["deg"] + 1) ** 2)
    sizes = [RESOLUTIONS[k % 4] for k in range(case["cams"])] if "cams" in case else [(case["w"], case["h"])]
    pixels = float(sum(w * h for w, h in sizes))
    project, composite = 400.0 * n * len(sizes), 21.0 * 70.0 * pixels
    forward = {"bytes": params + 12.0 * pixels, "flops": project + composite}
    if case["kind"] in ("call", "frame", "batch"):
        return forward
    backward = {"bytes": 2.0 * params + 12.0 * pixels, "flops": 2.0 * project + 3.0 * composite}
    if case["kind"] == "back":
        return backward
    total = {k: forward[k] + backward[k] for k in forward}
    if case["kind"] == "train":  # the target, and parameters and moments read and written
        total["bytes"] += 12.0 * pixels + 5.0 * params
        total["flops"] += 12.0 * params / 4.0
    return total


# ---- the same in float64 -------------------------------------------------------------------------


def _f32(v):
    return float(np.float32(v))


def _sh_basis(d, deg):
    """Real spherical harmonics with the Condon-Shortley phase, index l*l + l + m."""
    x, y, z = d.unbind(1)
    s = math.sqrt
    pi = math.pi
    Y = [torch.full_like(x, 0.5 / s(pi))]
    if deg >= 1:
        k = s(3 / (4 * pi))
        Y += [-k * y, k * z, -k * x]
    if deg >= 2:
        a, b, c = s(15 / pi) / 2, s(5 / pi) / 4, s(15 / pi) / 4
        Y += [a * x * y, -a * y * z, b * (2 * z * z - x * x - y * y), -a * x * z, c * (x * x - y * y)]
    if deg >= 3:
        a, b, c = s(35 / (2 * pi)) / 4, s(105 / pi) / 2, s(21 / (2 * pi)) / 4
        d0, e = s(7 / pi) / 4, s(105 / pi) / 4
        Y += [-a * y * (3 * x * x - y * y), b * x * y * z, -c * y * (4 * z * z - x * x - y * y),
              d0 * z * (2 * z * z - 3 * x * x - 3 * y * y), -c * x * (4 * z * z - x * x - y * y),
              e * z * (x * x - y * y), -a * x * (x * x - 3 * y * y)]
    return torch.stack(Y, 1)


def _project64(p, cam):
    """Per-Gaussian mean, covariance, opacity, colour and depth in float64
    (3DGS conventions), and which Gaussians are visible."""
    dev = p["means"].device
    V = torch.tensor(np.asarray(cam["viewmat"], np.float64), device=dev)
    fx, fy, cx, cy = (_f32(cam[k]) for k in ("fx", "fy", "cx", "cy"))
    t = p["means"] @ V[:3, :3].T + V[:3, 3]
    vis = t[:, 2] > _f32(cam["znear"])
    t = torch.where(vis[:, None], t, torch.tensor([0.0, 0.0, 1.0], dtype=t.dtype, device=dev))
    tx, ty, tz = t.unbind(1)
    lx, ly = 1.3 * _f32(cam["tan_fovx"]), 1.3 * _f32(cam["tan_fovy"])
    ux, uy = (tx / tz).clamp(-lx, lx), (ty / tz).clamp(-ly, ly)
    zero = torch.zeros_like(tz)
    J = torch.stack([fx / tz, zero, -fx * ux / tz, zero, fy / tz, -fy * uy / tz], 1).view(-1, 2, 3)
    w, x, y, z = (p["quats"] / p["quats"].norm(dim=1, keepdim=True)).unbind(1)
    Rm = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                      2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                      2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    A = (J @ V[:3, :3]) @ (Rm * p["scales"].exp()[:, None, :])
    S = A @ A.transpose(1, 2)
    s11, s12, s22 = S[:, 0, 0] + 0.3, S[:, 0, 1], S[:, 1, 1] + 0.3
    o = torch.sigmoid(p["opacities"])
    vis = vis & (o >= 1.0 / 255.0)
    d = p["means"] - torch.tensor(np.asarray(cam["campos"], np.float64), device=dev)
    Y = _sh_basis(d / d.norm(dim=1, keepdim=True), int(round(math.sqrt(p["sh"].shape[1]))) - 1)
    rgb = ((Y[:, :, None] * p["sh"]).sum(1) + 0.5).clamp(min=0.0)
    screen = torch.stack([fx * tx / tz + cx, fy * ty / tz + cy, s11, s12, s22, o], 1)
    return torch.cat([screen, rgb], 1), tz, vis


def _tile_lists64(q, tz, vis, W, H):
    """Gaussians by (tile, depth): the tiles of the 3-sigma square that the
    ellipse alpha = 1/255 can reach."""
    tiles_x, tiles_y = (W + 15) // 16, (H + 15) // 16
    mx, my, s11, s12, s22, o = q[:, :6].unbind(1)
    half = 0.5 * (s11 - s22)
    r3 = torch.ceil(3.0 * torch.sqrt(0.5 * (s11 + s22) + torch.sqrt((half * half + s12 * s12).clamp(min=0.1))))
    gam = 2.0 * torch.log(255.0 * o).clamp(min=0.0) * (1 + 1e-9) + 1e-9
    ex, ey = torch.sqrt(gam * s11) + 1e-6, torch.sqrt(gam * s22) + 1e-6

    def span(m, e, size):
        lo = torch.maximum(torch.ceil(m) - r3, torch.ceil(m - e)).clamp(min=0)
        hi = torch.minimum(torch.floor(m) + r3, torch.floor(m + e)).clamp(max=size - 1)
        # (tiles of the 3-sigma square; the reach only removes tiles without a contribution)
        return (lo / 16).floor().long(), (hi / 16).floor().long(), lo <= hi

    x0, x1, okx = span(mx, ex, W)
    y0, y1, oky = span(my, ey, H)
    # a tile of the square counts whole: extend back to tile borders is implied by the tile ids
    cnt = torch.where(vis & okx & oky, (x1 - x0 + 1) * (y1 - y0 + 1), torch.zeros_like(x0))
    order = torch.argsort(tz, stable=True)
    order = order[cnt[order] > 0]
    c = cnt[order]
    gid = torch.repeat_interleave(order, c)
    k = torch.arange(gid.numel(), device=q.device) - torch.repeat_interleave(torch.cumsum(c, 0) - c, c)
    wdt = (x1 - x0 + 1)[gid]
    tile = (y0[gid] + k // wdt) * tiles_x + x0[gid] + k % wdt
    del k, wdt
    tile, idx = torch.sort(tile.to(torch.int32), stable=True)
    gid = gid[idx].to(torch.int32)
    del idx
    bounds = torch.searchsorted(tile, torch.arange(tiles_x * tiles_y + 1, device=q.device, dtype=torch.int32))
    return gid, bounds


def _alpha64(e, px, py):
    """alpha of entries e [T, K, 9] at pixels [T, P]: [T, K, P]."""
    mx, my, s11, s12, s22, o = (v[..., None] for v in e[..., :6].unbind(-1))
    dx, dy = mx - px[:, None], my - py[:, None]
    power = -0.5 * (s22 * dx * dx - 2 * s12 * dx * dy + s11 * dy * dy) / (s11 * s22 - s12 * s12)
    a = (o * torch.exp(power)).clamp(max=0.99)
    return torch.where(a >= 1.0 / 255.0, a, torch.zeros_like(a))


def _composite64(q, gid, bounds, W, H, dL=None):
    """The image [3, H, W] over BG, and with dL the gradient of (image * dL)
    with respect to q."""
    dev = q.device
    tiles_x, tiles_y = (W + 15) // 16, (H + 15) // 16
    img = torch.zeros((3, tiles_y * 16, tiles_x * 16), dtype=torch.float64, device=dev)
    gq = torch.zeros_like(q) if dL is not None else None
    if dL is not None:
        full = torch.zeros_like(img)
        full[:, :H, :W] = dL
        dL = full
    bg = torch.tensor([_f32(v) for v in BG], dtype=torch.float64, device=dev)
    length = bounds[1:] - bounds[:-1]
    by_length = torch.argsort(length, descending=True)
    pix = torch.arange(256, device=dev)
    CHUNK = 128

    def gather(t, k0, k1):
        at = bounds[t][:, None] + torch.arange(k0, k1, device=dev)[None]
        have = at < bounds[t + 1][:, None]
        g = gid[at.clamp(max=max(0, gid.numel() - 1))].long()
        e = q[g]
        e[..., 5] = torch.where(have, e[..., 5], torch.zeros_like(e[..., 5]))  # opacity 0: never composited
        return e, g

    G = 64
    for i in range(0, by_length.numel(), G):
        t = by_length[i:i + G]
        most = int(length[t].max()) if gid.numel() else 0
        X = ((t % tiles_x) * 16)[:, None] + (pix % 16)[None]
        Yp = ((t // tiles_x) * 16)[:, None] + (pix // 16)[None]
        px, py = X.double(), Yp.double()
        T = torch.ones((t.numel(), 256), dtype=torch.float64, device=dev)
        T[(X >= W) | (Yp >= H)] = 0.0  # outside: stopped from the start
        Tout, C = T.clone(), torch.zeros((t.numel(), 256, 3), dtype=torch.float64, device=dev)
        walked = 0
        for k0 in range(0, most, CHUNK):
            e, _ = gather(t, k0, min(most, k0 + CHUNK))
            walked = min(most, k0 + CHUNK)
            a = _alpha64(e, px, py)
            after = T[:, None] * torch.cumprod(1 - a, 1)
            a = torch.where(after >= 1e-4, a, torch.zeros_like(a))  # the entry that would stop the pixel, and all behind it
            before = torch.cat([T[:, None], T[:, None] * torch.cumprod(1 - a, 1)], 1)
            C += torch.einsum("tkp,tkc->tpc", a * before[:, :-1], e[..., 6:])
            Tout = torch.where(T > 0, before[:, -1], Tout)
            T = torch.where(after[:, -1] >= 1e-4, before[:, -1], torch.zeros_like(T))
            if not bool((T > 0).any()):
                break
        img[:, Yp, X] = (C + Tout[..., None] * bg).permute(2, 0, 1)
        if dL is None or walked == 0:
            continue
        part = max(1, int(12_000_000 // (walked * 256)))
        for j in range(0, t.numel(), part):
            s = slice(j, j + part)
            e, g = gather(t[s], 0, walked)
            e.requires_grad_(True)
            a = _alpha64(e, px[s], py[s])
            inside = ((X[s] < W) & (Yp[s] < H))[:, None]
            with torch.no_grad():
                keep = (torch.cumprod(1 - a, 1) >= 1e-4) & inside
            a = torch.where(keep, a, torch.zeros_like(a))
            after = torch.exp(torch.cumsum(torch.log1p(-a), 1))
            before = torch.cat([torch.ones_like(after[:, :1]), after[:, :-1]], 1)
            Cg = torch.einsum("tkp,tkc->tpc", a * before, e[..., 6:]) + after[:, -1, :, None] * bg
            grad = dL[:, Yp[s], X[s]].permute(1, 2, 0) * inside[:, 0, :, None]
            ge, = torch.autograd.grad((Cg * grad).sum(), e)
            gq.index_add_(0, g.reshape(-1), ge.reshape(-1, 9))
    return img[:, :H, :W].contiguous(), gq


def _view64(p, cam, dL=None):
    """One view: the image, and with dL the gradients of the parameters p
    (dL may be a function of the image)."""
    with torch.set_grad_enabled(dL is not None):
        q, tz, vis = _project64(p, cam)
    with torch.no_grad():
        gid, bounds = _tile_lists64(q.detach(), tz.detach(), vis, cam["width"], cam["height"])
    if dL is None:
        return _composite64(q.detach(), gid, bounds, cam["width"], cam["height"])[0], None
    if callable(dL):
        dL = dL(_composite64(q.detach(), gid, bounds, cam["width"], cam["height"])[0])
    img, gq = _composite64(q.detach(), gid, bounds, cam["width"], cam["height"], dL.double())
    grads = torch.autograd.grad(q, [p[k] for k in KEYS], gq)
    return img, list(grads)


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    kind = case["kind"]
    if kind == "sort":
        keys, vals = _sort_input(case, seed, dev)
        # unsigned order: flip the sign bit of 64-bit keys
        flipped, idx = torch.sort(keys ^ (-(2 ** 63) if case["bits"] == 64 else 0), stable=True)
        return [keys[idx], vals[idx]]
    scene, cams = _scene(case, seed, dev), _cameras(case, seed)
    pixels = sum(c["width"] * c["height"] for c in cams)
    if kind in ("batch", "bgrad") and (pixels > 12_000_000 or case["n"] * len(cams) > 4_000_000):
        return None  # minutes in this form
    need = kind in ("grad", "back", "train", "bgrad")
    p = {k: scene[k].double().requires_grad_(need) for k in KEYS}
    shape = (3, cams[0]["height"], cams[0]["width"])
    if kind in ("call", "frame"):
        return _view64(p, cams[0])[0]
    if kind in ("grad", "back"):
        img, g = _view64(p, cams[0], _image_like(case, seed, "loss", shape, dev))
        return g if kind == "back" else [img, *g]
    if kind == "train":
        target = _image_like(case, seed, "target", shape, dev).double()
        scale = 1.0 / target.numel()
        img, g = _view64(p, cams[0], lambda im: torch.sign(im - target) * scale)
        m, v = _moments(scene, seed, dev)
        t = RESUMED_AT + 1
        new = []
        for k, gk in zip(KEYS, g):
            mk = BETAS[0] * m[k].double() + (1 - BETAS[0]) * gk
            vk = BETAS[1] * v[k].double() + (1 - BETAS[1]) * gk * gk
            new.append(p[k].detach() - LR[k] * (mk / (1 - BETAS[0] ** t)) / ((vk / (1 - BETAS[1] ** t)).sqrt() + EPS))
        return [((img - target).abs().sum() * scale), img, *g, *new]
    images, total, at = [], None, 0
    flat = _image_like(case, seed, "loss", (3 * pixels,), dev) if kind == "bgrad" else None
    for cam in cams:
        size = 3 * cam["width"] * cam["height"]
        dL = flat[at:at + size].view(3, cam["height"], cam["width"]) if flat is not None else None
        img, g = _view64(p, cam, dL)
        images.append(img.reshape(-1))
        at += size
        if g is not None:
            total = g if total is None else [a + b for a, b in zip(total, g)]
    images = torch.cat(images)
    return images if kind == "batch" else [images, *total]
