"""The calls a user of the point rasterizer makes, over the range of sizes they are made at.

Every case goes through the public entry points of ``paper_2508_19140_gb300.rast``: the
C-ABI calls on a workspace that the program keeps (``rasterize_fwd``, ``rasterize_batch``,
``rasterize_clouds``), the autograd calls (``rasterize``, ``rasterize_views``), the background
composite and the contraction. Point clouds are the clustered mixture of
``paper_2508_19140_gb300/scenes.py`` (64 anisotropic Gaussian clusters and a 10 % uniform
background, in random order), drawn on the GPU; the work splits (tile edge, blend depth, record
copy) are the ones the autotuner picks for the workloads of ``bench.py``.
"""
import math

import torch

from paper_2508_19140_gb300 import rast, scenes

DEV = "cuda"
T_MIN, ALPHA_MAX, DILATION = 1e-4, 0.99, 0.16


def listed():
    return [
        # a thumbnail or unit-test sized frame: the smallest call, where launches and latency count
        {"name": "thumb_fwd_20k", "kind": "fwd", "n": 20000, "w": 128, "h": 128, "c": 4, "bf16": False,
         "gauss": False, "tile": 16},
        # one step of a small training run through autograd, odd image, three channels
        {"name": "autograd_60k_c3", "kind": "autograd", "n": 60001, "w": 301, "h": 203, "c": 3, "bf16": False,
         "gauss": False, "tile": 16},
        # a medium preview frame under no_grad, ragged size, eight BF16 channels
        {"name": "preview_500k_c8_bf16", "kind": "nograd", "n": 500009, "w": 799, "h": 601, "c": 8, "bf16": True,
         "gauss": False, "tile": 16},
        # a training step over three uneven views at once through autograd, BF16 features
        {"name": "autograd_3views_bf16", "kind": "autograd", "views": 3, "n": 400000, "w": 641, "h": 479, "c": 4,
         "bf16": True, "gauss": False, "tile": 16},
        # the training-shape step: 4 M points at 1280x832, forward and backward on a kept workspace
        {"name": "train_4M", "kind": "step", "n": 1 << 22, "w": 1280, "h": 832, "c": 4, "bf16": False,
         "gauss": False, "tile": 8},
        # the inference frame: 32 M points at 1920x1080
        {"name": "infer_32M", "kind": "fwd", "n": 1 << 25, "w": 1920, "h": 1080, "c": 4, "bf16": False,
         "gauss": False, "tile": 16},
        # interactive viewing with points as small Gaussians, forward only, odd size
        {"name": "gauss_view_2M", "kind": "fwd", "n": 2000003, "w": 1599, "h": 899, "c": 4, "bf16": False,
         "gauss": True, "tile": 16},
        # training with points as small Gaussians: gradients to features, opacity, positions and scales
        {"name": "gauss_train_16M_bf16", "kind": "step", "n": 1 << 24, "w": 1920, "h": 1080, "c": 4, "bf16": True,
         "gauss": True, "tile": 16},
        # a training batch of eight uneven views, 640x480 to 1920x1080, 1 M to 16 M points each, in one call
        {"name": "batch_8views_bf16", "kind": "step", "views": 8, "n": 1 << 24, "w": 1920, "h": 1080, "c": 8,
         "bf16": True, "gauss": False, "tile": 8, "copy": True},
        # the ring buffer of view-specific clouds: four clouds rendered into one image
        {"name": "ring_4x2M", "kind": "clouds", "views": 4, "n": 2000001, "w": 1280, "h": 720, "c": 4, "bf16": False,
         "gauss": False, "tile": 16},
        # the distilled background behind a training frame, forward and backward
        {"name": "background_1280x832", "kind": "background", "w": 1280, "h": 832, "c": 4, "mh": 1024, "mw": 2048},
        # the spherical contraction of sampled positions before the appearance field
        {"name": "contract_8M", "kind": "contract", "n": 8000003},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fwd", "fwd", "step", "step", "nograd", "autograd", "clouds", "background", "contract"])
    if kind == "contract":
        return {"kind": kind, "n": _log_int(rng, 1000, 32 << 20)}
    w = _log_int(rng, 97, 1920)
    h = max(64, min(1080, int(w * rng.uniform(0.55, 0.8))))
    if kind == "background":
        mh = rng.choice([128, 512, 1024])
        return {"kind": kind, "w": w, "h": h, "c": rng.choice([3, 4, 8]), "mh": mh, "mw": 2 * mh}
    gauss = rng.random() < 0.35
    views = {"clouds": rng.randint(2, 5), "step": rng.choice([1, 1, 3]), "autograd": rng.choice([1, 1, 2])}.get(kind, 1)
    top = {"fwd": 16e6, "step": 8e6, "nograd": 4e6, "autograd": 2e6, "clouds": 8e6}[kind] / views
    # between a quarter point and sixteen points a pixel, as the listed frames have
    n = min(int(top), max(5000, int(w * h * math.exp(rng.uniform(math.log(0.25), math.log(16.0))))))
    case = {"kind": kind, "n": n, "w": w, "h": h, "c": rng.choice([1, 2, 3, 4, 4, 4, 8, 16]),
            "bf16": rng.random() < 0.4, "gauss": gauss, "tile": rng.choice([16, 16, 8])}
    if views > 1:
        case["views"] = views
    if kind == "step" and not gauss and rng.random() < 0.5:
        case["copy"] = True
    return case


# ------------------------------------------------------------------ inputs

def _cameras(case):
    """(camera, points) of every view; the views of a batch are uneven."""
    w, h, n, k = case["w"], case["h"], case["n"], case.get("views", 1)
    if case["kind"] == "clouds":
        cam = scenes.orbit_camera(w, h, 6.0, 30.0, 15.0)
        return [(cam, max(1, n - 1001 * i)) for i in range(k)]
    if case["gauss"]:
        f = 1000.0 * w / 1920.0
        return [(scenes.orbit_camera(w, h, 5.0, 20.0 + 45.0 * i, 10.0, f), n) for i in range(k)]
    if k == 8:
        return [(scenes.orbit_camera(vw, vh, 6.0, 45.0 * i, 15.0), vn)
                for i, (vw, vh, vn) in enumerate(scenes.BATCH_VIEWS)]
    shrink = [1.0, 0.75, 0.5, 0.6, 0.9]
    return [(scenes.orbit_camera(max(8, int(w * shrink[i])), max(8, int(h * shrink[i])), 6.0, 30.0 + 45.0 * i, 15.0),
             max(1, int(n * shrink[i]))) for i in range(k)]


def _clustered(g, n):
    """The clustered mixture of scenes.clustered_points, drawn on the GPU."""
    k = 64
    centres = torch.rand((k, 3), generator=g, device=DEV) * 3.0 - 1.5
    sig = 0.02 + 0.28 * torch.rand((k, 3), generator=g, device=DEV)
    rot, _ = torch.linalg.qr(torch.randn((k, 3, 3), generator=g, device=DEV))
    basis = rot * sig[:, None, :]
    which = torch.randint(0, k, (n,), generator=g, device=DEV)
    local = torch.randn((n, 3), generator=g, device=DEV)
    out = torch.empty((n, 3), device=DEV)
    step = 1 << 22  # in pieces: the gathered bases are nine floats a point
    for a in range(0, n, step):
        b = min(n, a + step)
        out[a:b] = (basis[which[a:b]] * local[a:b, None, :]).sum(-1) + centres[which[a:b]]
    bg = torch.rand((n,), generator=g, device=DEV) < 0.10
    out[bg] = torch.rand((n, 3), generator=g, device=DEV)[bg] * 4.0 - 2.0
    return out


def _gauss_points(g, cam, n):
    """Clustered points kept to view depths of 1.9 to 10, as scenes.gaussian_view has them."""
    r = torch.tensor(cam.R[2], device=DEV)
    have, got = 0, []
    while have < n:
        p = _clustered(g, max(n // 2, 4096))
        z = p @ r + float(cam.t[2])
        p = p[(z >= 1.9) & (z <= 10.0)]
        got.append(p)
        have += len(p)
    return torch.cat(got)[:n].contiguous()


def _opacity(g, n):
    """Beta(2, 2): the middle of three uniforms."""
    return torch.rand((n, 3), generator=g, device=DEV).median(dim=1).values


def _views(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    c, out = case["c"], []
    for cam, n in _cameras(case):
        xyz = _gauss_points(g, cam, n) if case["gauss"] else _clustered(g, n)
        op = _opacity(g, n)
        feat = torch.rand((n, c), generator=g, device=DEV)
        if case["bf16"]:
            feat = feat.to(torch.bfloat16)
        scale = None
        if case["gauss"]:
            scale = torch.exp(torch.empty(n, device=DEV).uniform_(math.log(1e-3), math.log(1e-2), generator=g))
        v = {"cam": cam, "xyz": xyz, "op": op, "feat": feat, "scale": scale}
        if case["kind"] in ("step", "autograd"):
            v["g"] = [torch.randn(s, generator=g, device=DEV)
                      for s in ((cam.height, cam.width, c), (cam.height, cam.width), (cam.height, cam.width))]
        out.append(v)
    return out


def _image(cam, c):
    return [torch.empty(s, device=DEV) for s in ((cam.height, cam.width, c), (cam.height, cam.width),
                                                 (cam.height, cam.width))]


def _mode(case):
    return "gaussian" if case["gauss"] else "bilinear"


def _world_positions(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    n = case["n"]  # most samples inside the unit ball, a long tail outside
    return torch.randn((n, 3), generator=g, device=DEV) * torch.exp(torch.randn((n, 1), generator=g, device=DEV))


def _background(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    w, h, c = case["w"], case["h"], case["c"]
    lam = (torch.arange(case["mw"], device=DEV) + 0.5) / case["mw"] * (2 * math.pi) - math.pi
    th = (torch.arange(case["mh"], device=DEV) + 0.5) / case["mh"] * math.pi
    ph = torch.rand((3, c), generator=g, device=DEV) * (2 * math.pi)
    env = (0.5 + 0.25 * torch.cos(th[:, None, None] + ph[0])
           + 0.1 * torch.cos(lam[None, :, None] + ph[1]) * torch.sin(th)[:, None, None]
           + 0.05 * torch.cos(2 * lam[None, :, None] + th[:, None, None] + ph[2])).contiguous()
    return {"cam": scenes.orbit_camera(w, h, 6.0, 30.0, 15.0), "env": env,
            "feat": torch.rand((h, w, c), generator=g, device=DEV),
            "alpha": torch.rand((h, w), generator=g, device=DEV),
            "g": torch.randn((h, w, c), generator=g, device=DEV),
            "ga": torch.randn((h, w), generator=g, device=DEV)}


# ------------------------------------------------------------------ state and passes

def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    if kind == "contract":
        s["xyz"] = _world_positions(case, seed)
        s["out"] = torch.empty_like(s["xyz"])
        return s
    if kind == "background":
        b = _background(case, seed)
        s.update(b)
        s["c_cam"], s["c_env"] = rast.make_camera(b["cam"]), rast.make_envmap(b["env"])
        s["dirs"] = torch.empty((case["h"], case["w"], 3), device=DEV)
        rast.rasterize_view_dirs(s["c_cam"], s["dirs"])  # cached over frames: they depend on the intrinsics only
        s["out"], s["d_map"] = torch.empty_like(b["feat"]), torch.empty_like(b["env"])
        s["g_alpha"] = torch.empty_like(b["ga"])
        s["scratch"] = torch.empty(rast.rasterize_bg_scratch_size(s["c_env"]), dtype=torch.uint8, device=DEV)
        return s
    views = _views(case, seed)
    s["views"] = views
    if kind in ("autograd", "nograd"):
        s["kw"] = dict(mode=_mode(case), tile=case["tile"])
        s["items"] = [(v["xyz"], v["op"], v["feat"], v["cam"], v["scale"]) for v in views]
        if kind == "autograd":
            s["leaves"] = []
            for v in views:
                v["op"].requires_grad_(True)
                v["feat"].requires_grad_(True)
                s["leaves"] += [v["feat"], v["op"]]
                if case["gauss"]:
                    v["xyz"].requires_grad_(True)
                    v["scale"].requires_grad_(True)
                    s["leaves"] += [v["xyz"], v["scale"]]
            s["grads"] = [t for v in views for t in v["g"]]
        return s
    opts = rast.make_opts(mode=_mode(case), tile=case["tile"],
                          flags=rast.FLAG_SAVE_FOR_BWD if case.get("copy") else 0)
    s["opts"] = opts
    s["pts"] = [rast.make_points(v["xyz"], v["op"], v["feat"], v["scale"]) for v in views]
    if kind in ("fwd", "clouds"):
        cam = views[0]["cam"]
        s["cam"] = rast.make_camera(cam)
        s["out"] = _image(cam, case["c"])
        s["im"] = rast.make_images(*s["out"])
        if kind == "clouds":
            size = rast.rasterize_clouds_workspace_size(s["pts"], s["cam"], opts)
        else:
            v = rast.View()
            v.pts, v.cam, v.out = s["pts"][0], s["cam"], s["im"]
            size = rast.rasterize_workspace_size([v], opts)
    else:
        s["out"], s["cviews"] = [], []
        for v, p in zip(views, s["pts"]):
            n, c = v["feat"].shape
            im = _image(v["cam"], c)
            d = [torch.empty((n, c), device=DEV), torch.empty((n,), device=DEV)]
            if case["gauss"]:
                d += [torch.empty((n, 3), device=DEV), torch.empty((n,), device=DEV)]
            cv = rast.View()
            cv.pts, cv.cam, cv.out = p, rast.make_camera(v["cam"]), rast.make_images(*im)
            cv.grad = rast.make_grads(*v["g"], *d)
            s["cviews"].append(cv)
            s["out"] += im + d
        size = rast.rasterize_workspace_size(s["cviews"], opts)
    s["ws"] = torch.empty(size, dtype=torch.uint8, device=DEV)
    return s


def run(s):
    kind = s["kind"]
    if kind == "fwd":
        rast.rasterize_fwd(s["pts"][0], s["cam"], s["opts"], s["ws"], s["im"])
        return s["out"]
    if kind == "step":
        rast.rasterize_batch(s["cviews"], rast.PASS_FWD | rast.PASS_BWD, s["opts"], s["ws"])
        return s["out"]
    if kind == "clouds":
        rast.rasterize_clouds(s["pts"], None, s["cam"], s["im"], rast.PASS_FWD, s["opts"], s["ws"])
        return s["out"]
    if kind == "nograd":
        with torch.no_grad():
            xyz, op, feat, cam, scale = s["items"][0]
            return list(rast.rasterize(xyz, op, feat, cam, scale, **s["kw"]))
    if kind == "autograd":
        images = [t for im in rast.rasterize_views(s["items"], **s["kw"]) for t in im]
        grads = torch.autograd.grad(images, s["leaves"], s["grads"])
        return [t.detach() for t in images] + list(grads)
    if kind == "background":
        rast.rasterize_bg_composite(s["c_cam"], s["c_env"], s["dirs"], s["feat"], s["alpha"], s["out"])
        s["g_alpha"].copy_(s["ga"])  # the loss's own dL/dalpha, which the call adds to
        rast.rasterize_bg_composite_bwd(s["c_cam"], s["c_env"], s["dirs"], s["alpha"], s["g"], s["g_alpha"],
                                        s["d_map"], s["scratch"])
        return [s["out"], s["g_alpha"], s["d_map"]]
    rast.rasterize_contract(s["xyz"], s["out"])
    return s["out"]


def work(case):
    """Every input read once and every output written once; operations of the projection (about 40
    a point) and of four blended fragments a point."""
    kind = case["kind"]
    if kind == "contract":
        return {"bytes": 24.0 * case["n"], "flops": 15.0 * case["n"]}
    if kind == "background":
        px, c, m = case["w"] * case["h"], case["c"], case["mh"] * case["mw"] * case["c"]
        # forward: directions, features, alpha, map in, image out; backward: directions, alpha, the
        # image's and alpha's gradients, map in, alpha's and the map's gradients out
        return {"bytes": 4.0 * (px * (3 + 2 * c + 1) + m + px * (3 + 1 + c + 2) + 2 * m),
                "flops": px * (60.0 + 24.0 * c)}
    c, fb = case["c"], 2 if case["bf16"] else 4
    cams = _cameras(case)
    n = sum(k for _, k in cams)
    px = sum(cam.width * cam.height for cam, _ in (cams[:1] if kind == "clouds" else cams))
    by = n * (16 + fb * c + (4 if case["gauss"] else 0)) + px * 4 * (c + 2)
    fl = n * (40.0 + 4 * (2 * c + 6))
    if kind in ("step", "autograd"):
        by += px * 4 * (c + 2) + n * (4 + (4 if kind == "step" else fb) * c + (16 if case["gauss"] else 0))
        fl += n * 4 * (4.0 * c + 12)
    return {"bytes": float(by), "flops": float(fl)}


# ------------------------------------------------------------------ the same in 64 bits

def _project(v, gauss, leaves=None):
    """Screen positions, depths (and conics, radii) in FP32, one rounded operation at a time in the order the
    header's conventions give; with `leaves` (xyz, scale in FP64) the same in FP64, for the chain rule."""
    cam = v["cam"]
    dt = torch.float32 if leaves is None else torch.float64
    xyz, s = (v["xyz"].detach(), v["scale"]) if leaves is None else leaves
    k = lambda a: torch.tensor(float(a), dtype=torch.float32, device=DEV).to(dt)  # noqa: E731
    x, y, z = xyz[:, 0], xyz[:, 1], xyz[:, 2]
    row = lambda i: k(cam.R[i][0]) * x + k(cam.R[i][1]) * y + k(cam.R[i][2]) * z + k(cam.t[i])  # noqa: E731
    xc, yc, zc = row(0), row(1), row(2)
    fx, fy = k(cam.fx), k(cam.fy)
    u, w = fx * (xc / zc) + k(cam.cx), fy * (yc / zc) + k(cam.cy)
    if not gauss:
        return u, w, zc
    s = s.detach() if leaves is None else s
    s2, zz = s * s, zc * zc
    j00, j11, j02, j12 = fx / zc, fy / zc, -(fx * xc / zz), -(fy * yc / zz)
    s00 = s2 * (j00 * j00 + j02 * j02) + k(DILATION)
    s01 = s2 * (j02 * j12)
    s11 = s2 * (j11 * j11 + j12 * j12) + k(DILATION)
    det = s00 * s11 - s01 * s01
    hd = 0.5 * (s00 - s11)
    r = torch.ceil(3.0 * torch.sqrt(0.5 * (s00 + s11) + torch.sqrt(hd * hd + s01 * s01)))
    return u, w, zc, s11 / det, -s01 / det, s00 / det, r


def _fragments(proj, cam, op, gauss):
    """Per fragment: point, pixel, the FP32 alpha that decides, the FP64 alpha, the FP64 weight and whether the
    alpha is clamped; in (depth, point) order of the points."""
    w, h = cam.width, cam.height
    u, v, z = proj[:3]
    near = torch.tensor(cam.near, dtype=torch.float32, device=DEV)
    far = torch.tensor(cam.far, dtype=torch.float32, device=DEV)
    um, vm = u - 0.5, v - 0.5
    vis = (z > near) & (z < far)
    if gauss:
        r = proj[6]
        x0, x1 = torch.ceil(um - r).clamp(min=0), torch.floor(um + r).clamp(max=w - 1)
        y0, y1 = torch.ceil(vm - r).clamp(min=0), torch.floor(vm + r).clamp(max=h - 1)
    else:
        fi, fj = torch.floor(um), torch.floor(vm)
        vis &= (fi >= -1) & (fi <= w - 1) & (fj >= -1) & (fj <= h - 1)
        x0, x1, y0, y1 = fi, fi + 1, fj, fj + 1
    vis &= (x0 <= x1) & (y0 <= y1)
    idx = torch.nonzero(vis).squeeze(1)
    idx = idx[torch.sort(z[idx], stable=True).indices]
    out = []
    step = 1 << (19 if gauss else 22)
    amax = torch.tensor(ALPHA_MAX, dtype=torch.float32, device=DEV)
    for a in range(0, len(idx), step):
        p = idx[a:a + step]
        bx, by = x0[p].long(), y0[p].long()
        bw, bh = x1[p].long() - bx + 1, y1[p].long() - by + 1
        cnt = bw * bh
        rep = torch.repeat_interleave(torch.arange(len(p), device=DEV), cnt)
        k = torch.arange(len(rep), device=DEV) - (torch.cumsum(cnt, 0) - cnt)[rep]
        px, py = bx[rep] + k % bw[rep], by[rep] + k // bw[rep]
        q = p[rep]
        ok = (px >= 0) & (px < w) & (py >= 0) & (py < h)
        if gauss:
            dx, dy = px.float() - um[q], py.float() - vm[q]
            ca, cb, cc = proj[3][q], proj[4][q], proj[5][q]
            t = cb * dx * dy
            m = ca * dx * dx + (t + t) + cc * dy * dy
            ok &= m <= 9.0
            dx, dy = dx[ok].double(), dy[ok].double()
            wt32 = torch.exp(-0.5 * m[ok])
            wt = torch.exp(-0.5 * (ca[ok].double() * dx * dx + 2 * cb[ok].double() * dx * dy
                                   + cc[ok].double() * dy * dy))
        else:
            fa, fb = um - fi, vm - fj
            q0 = q[ok]
            left, top = (px == bx[rep])[ok], (py == by[rep])[ok]
            ax, by_ = fa[q0], fb[q0]
            wt32 = torch.where(left, 1 - ax, ax) * torch.where(top, 1 - by_, by_)
            ax, by_ = ax.double(), by_.double()
            wt = torch.where(left, 1 - ax, ax) * torch.where(top, 1 - by_, by_)
        q = q[ok]
        o32 = op[q] * wt32
        raw = op[q].double() * wt
        out.append((q.int(), (py * w + px)[ok].int(), torch.minimum(o32, amax), raw.clamp(max=float(amax)), wt,
                    o32 > amax))
    return [torch.cat(t) for t in zip(*out)]


def _exact_image(clouds, cam, c, gauss, grads=None):
    """Images of one camera's clouds (concatenated), and with `grads` the points' gradients, in FP64; the
    discrete decisions (order, coverage, termination) in FP32."""
    cat = lambda k: torch.cat([v[k].detach() for v in clouds]) if clouds[0][k] is not None else None  # noqa: E731
    v = {"cam": cam, "xyz": cat("xyz"), "scale": cat("scale")}
    op, feat = cat("op"), cat("feat")
    n, px = len(op), cam.width * cam.height
    proj = _project(v, gauss)
    pt, pix, a32, a64, wt, clamped = _fragments(proj, cam, op, gauss)
    pix, order = torch.sort(pix, stable=True)
    pt, a32, a64 = pt[order], a32[order], a64[order]
    if grads is not None:
        wt, clamped = wt[order], clamped[order]
    del order
    cnt = torch.bincount(pix.long(), minlength=px)
    del pix
    start = torch.cumsum(cnt, 0) - cnt
    tmin = torch.tensor(T_MIN, dtype=torch.float32, device=DEV)
    F = torch.zeros((px, c), dtype=torch.float64, device=DEV)
    A, D = torch.zeros(px, dtype=torch.float64, device=DEV), torch.zeros(px, dtype=torch.float64, device=DEV)
    act = torch.nonzero(cnt > 0).squeeze(1)
    T32, T64 = torch.ones(len(act), device=DEV), torch.ones(len(act), dtype=torch.float64, device=DEV)
    Tfin = torch.ones(px, dtype=torch.float64, device=DEV)
    layers, k = [], 0
    while len(act):  # the k-th fragment of every pixel that still blends
        i = start[act] + k
        nxt = T32 * (1 - a32[i])
        go = nxt >= tmin
        act, i, T32, T64 = act[go], i[go], nxt[go], T64[go]
        a, q = a64[i], pt[i].long()
        wgt = T64 * a
        F[act] += wgt[:, None] * feat[q].double()
        A[act] += wgt
        D[act] += wgt * proj[2][q].double()
        if grads is not None:
            layers.append((act, i, T64))
        T64 = T64 * (1 - a)
        Tfin[act] = T64
        k += 1
        more = cnt[act] > k
        act, T32, T64 = act[more], T32[more], T64[more]
    images = [F.view(cam.height, cam.width, c), A.view(cam.height, cam.width), D.view(cam.height, cam.width)]
    if grads is None:
        return images, None
    gF, gA, gD = grads[0].reshape(px, c).double(), grads[1].reshape(px).double(), grads[2].reshape(px).double()
    S = torch.zeros(px, dtype=torch.float64, device=DEV)  # what lies behind, with its gradient
    d_feat = torch.zeros((n, c), dtype=torch.float64, device=DEV)
    d_op = torch.zeros(n, dtype=torch.float64, device=DEV)
    d_geo = torch.zeros((n, 6), dtype=torch.float64, device=DEV) if gauss else None  # u, v, a, b, c, z
    for act, i, T in reversed(layers):
        a, q = a64[i], pt[i].long()
        gf, gd = gF[act], gD[act]
        e = (gf * feat[q].double()).sum(1) + gd * proj[2][q].double()
        da = T * e - (S[act] - gA[act] * Tfin[act]) / (1 - a)
        wgt = T * a
        S[act] += wgt * e
        d_feat.index_add_(0, q, wgt[:, None] * gf)
        da = torch.where(clamped[i], torch.zeros_like(da), da)
        d_op.index_add_(0, q, wt[i] * da)
        if gauss:
            dx = (act % cam.width).double() - (proj[0][q] - 0.5).double()
            dy = (act // cam.width).double() - (proj[1][q] - 0.5).double()
            ca, cb, cc = (proj[j][q].double() for j in (3, 4, 5))
            dm = -0.5 * op[q].double() * wt[i] * da
            d_geo.index_add_(0, q, torch.stack([-dm * (2 * ca * dx + 2 * cb * dy), -dm * (2 * cb * dx + 2 * cc * dy),
                                                dm * dx * dx, 2 * dm * dx * dy, dm * dy * dy, wgt * gd], 1))
    points = [d_feat, d_op]
    if gauss:
        xyz, s = v["xyz"].double().requires_grad_(True), v["scale"].double().requires_grad_(True)
        hit = (d_geo != 0).any(1)
        with torch.enable_grad():
            p = _project(v, True, (xyz, s))
            loss = sum((torch.where(hit, p[j], torch.zeros_like(p[j])) * d_geo[:, g]).sum()
                       for g, j in enumerate((0, 1, 3, 4, 5, 2)))
            points += list(torch.autograd.grad(loss, (xyz, s)))
    return images, points


@torch.no_grad()
def exact(case, seed):
    kind = case["kind"]
    if kind == "contract":
        x = _world_positions(case, seed).double()
        r = x.norm(dim=1, keepdim=True)
        return torch.where(r <= 1, x, (2 - 1 / r) * x / r)
    if kind == "background":
        return _exact_background(case, seed)
    views = _views(case, seed)
    if kind == "clouds":
        return _exact_image(views, views[0]["cam"], case["c"], case["gauss"])[0]
    got = [_exact_image([v], v["cam"], case["c"], case["gauss"], v.get("g")) for v in views]
    if kind == "step":
        return [t for im, p in got for t in im + p]
    if kind == "autograd":
        return [t for im, _ in got for t in im] + [t for _, p in got for t in p]
    return got[0][0]


def _exact_background(case, seed):
    b = _background(case, seed)
    cam, w, h, c, mw, mh = b["cam"], case["w"], case["h"], case["c"], case["mw"], case["mh"]
    R = torch.tensor(cam.R, device=DEV).double()
    f32 = lambda a: float(torch.tensor(float(a)).float())  # noqa: E731
    x = (torch.arange(w, device=DEV).double() + 0.5 - f32(cam.cx)) / f32(cam.fx)
    y = (torch.arange(h, device=DEV).double() + 0.5 - f32(cam.cy)) / f32(cam.fy)
    d = torch.stack([x[None, :].expand(h, w), y[:, None].expand(h, w), torch.ones((h, w), device=DEV).double()], -1)
    d = (d / d.norm(dim=-1, keepdim=True)) @ R
    X = (torch.atan2(d[..., 0], d[..., 2]) / (2 * math.pi) + 0.5) * mw - 0.5
    Y = torch.acos(d[..., 1].clamp(-1, 1)) / math.pi * mh - 0.5
    x0, y0 = torch.floor(X), torch.floor(Y)
    fa, fb = X - x0, Y - y0
    env, alpha, g = b["env"].double().view(-1, c), b["alpha"].double(), b["g"].double()
    bg = torch.zeros((h, w, c), dtype=torch.float64, device=DEV)
    d_map = torch.zeros((mh * mw, c), dtype=torch.float64, device=DEV)
    for j, wy in ((0, 1 - fb), (1, fb)):
        for i, wx in ((0, 1 - fa), (1, fa)):
            t = (y0.long() + j).clamp(0, mh - 1) * mw + (x0.long() + i) % mw
            wt = (wx * wy)[..., None]
            bg += wt * env[t]
            d_map.index_add_(0, t.view(-1), (wt * (1 - alpha)[..., None] * g).view(-1, c))
    return [b["feat"].double() + (1 - alpha)[..., None] * bg, b["ga"].double() - (g * bg).sum(-1),
            d_map.view(mh, mw, c)]
