"""The work a user of the ray caster has it do, as timed cases.

Each case is one request (or one small group of requests that belong together) made through
the package's public entry points: renders of one view of a cube, moment maps, in-ray
smoothing, the separable smoothing, a batch of sub-cubes, a training step on the compositing
render.  ``listed()`` names the fixed cases, ``draw(rng)`` gives more of the same ranges,
``prepare`` makes the inputs on the GPU, ``run`` is one pass, ``work`` the bytes and
operations a pass cannot do without and ``exact`` the outputs in 64 bits from plain torch.
"""
from __future__ import annotations

import math
import random
from types import SimpleNamespace

import numpy as np
import torch

import paper_1707_00442_gb300 as shw

DEV = "cuda"

# Colour-map domains and transfer-function settings of the repository's own workloads, in units
# of the noise sigma (cubes of noise and sources), and for cubes of U[0,1] voxels.
NOISE = dict(lo=-3.0, hi=8.0)
UNIT = dict(lo=0.0, hi=1.0)
RATIO = dict(lo=0.0, hi=1.0, ratio_floor=1.0)


def _render(name, nx, ny, nz, width, height, mode, **more):
    c = dict(kind="render", nx=nx, ny=ny, nz=nz, width=width, height=height, mode=mode, data="sources", storage="f32",
             interp="trilinear", axis_view=False, yaw=30.0, pitch=20.0, ortho=False, step=0.5, opacity_scale=1.0,
             clip=False, smooth="none", smooth_size=0, outputs="image", **(RATIO if mode == "ratio" else NOISE))
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # The smallest call: the peak map of a cut-out around one source, every output taken.
        _render("cutout_map", 64, 64, 64, 128, 128, "mip", axis_view=True, outputs="all"),
        # An integral-field galaxy (two lines in two separate small cubes of odd sizes), its
        # line ratio while the view is turned.
        _render("ifu_ratio", 50, 50, 37, 1000, 1000, "ratio", storage="two", yaw=70.0, outputs="image"),
        # An interferometer mosaic: rows of 750 floats (no 16-byte multiple) and NaN outside the
        # footprint, composited.
        _render("mosaic_composite", 750, 750, 70, 1000, 1000, "composite", data="mosaic", yaw=20.0,
                opacity_scale=0.05),
        # The paper's benchmark cube without interpolation: nearest voxels, the peak and its
        # channel read back as well.
        _render("uniform_nearest", 512, 512, 512, 1000, 1000, "mip", data="uniform", interp="nearest", yaw=120.0,
                outputs="all", **UNIT),
        # The frame of an interactive session on a survey cube at full HD.
        _render("survey_composite", 512, 512, 1024, 1920, 1080, "composite", opacity_scale=0.01),
        # Two lines of a survey field kept in half the memory: pack the pair to binary16, then
        # render their ratio.
        _render("survey_ratio_f16", 512, 512, 1024, 1920, 1080, "ratio", storage="f16_linear"),
        # Moment maps of the survey cube down the spectral axis: the peak with its channel and
        # the intensity-weighted mean channel.
        dict(name="survey_moment_maps", kind="maps", nx=512, ny=512, nz=1024, width=512, height=512, step=0.5, **NOISE),
        # In-shader smoothing of the paper's benchmark: the 9-tap Gaussian on each axis ...
        _render("inray_gauss9", 512, 512, 512, 1000, 1000, "mip", data="uniform", smooth="gauss", smooth_size=9,
                yaw=120.0, **UNIT),
        # ... and the box along the ray.
        _render("inray_box5", 512, 512, 512, 1000, 1000, "mip", data="uniform", smooth="box", smooth_size=5,
                yaw=120.0, **UNIT),
        # The separable smoothing of a whole survey cube before it is rendered.
        dict(name="survey_smooth", kind="smooth", nx=512, ny=512, nz=1024, sigma=2.0, radius=6, pair=False),
        # Postage stamps of the detected galaxies: one batch plan, half of the sub-cubes float32
        # and half packed to bfloat16 bricks by the user.
        dict(name="stamps_batch", kind="batch", count=400, lo_dim=32, hi_dim=256, size=256, layout=1, bricks="half",
             step=0.5, opacity_scale=0.02, **NOISE),
        # One step of fitting a cube, a colour map and an opacity to a target image.
        dict(name="fit_step", kind="fit", nx=256, ny=256, nz=256, width=512, height=512, yaw=30.0, pitch=20.0, step=0.5,
             opacity_scale=0.02, ckpt_interval=64, **NOISE),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choices(["render", "inray", "maps", "smooth", "batch", "fit"], [46, 14, 8, 14, 9, 9])[0]
    if kind in ("render", "inray"):
        top = 640 if kind == "render" else 320
        nx, ny, nz = (_logint(rng, 32, top) for _ in range(3))
        if rng.random() < 0.3:
            nx = (nx + 3) // 4 * 4
        width, height = _logint(rng, 96, 1600), _logint(rng, 96, 1200)
        data = rng.choice(["sources", "uniform", "mosaic"])
        dom = UNIT if data == "uniform" else NOISE
        more = dict(data=data, yaw=round(rng.uniform(0, 360), 2), pitch=round(rng.uniform(-70, 70), 2),
                    ortho=rng.random() < 0.25, step=rng.choice([0.5, 0.5, 0.5, 1.0, 0.37]),
                    interp="nearest" if rng.random() < 0.25 else "trilinear",
                    outputs=rng.choice(["image", "image", "all"]), opacity_scale=rng.choice([0.01, 0.05, 0.22]), **dom)
        if kind == "inray":
            width, height = min(width, 1000), min(height, 800)
            more.update(smooth=rng.choice(["box", "gauss"]))
            more.update(smooth_size=rng.choice([3, 5, 7, 9] if more["smooth"] == "box" else [5, 9, 13]),
                        step=0.5 if rng.random() < 0.8 else 1.0, interp="trilinear")
            return _render("", nx, ny, nz, width, height, rng.choice(["mip", "avg", "composite"]), **more)
        mode = rng.choice(["mip", "avg", "composite", "composite", "spectral", "ratio", "moment1"])
        if mode == "ratio":
            more.update(storage=rng.choice(["two", "pair", "f16_linear", "bf16"]), data="sources", **RATIO)
        else:
            more.update(storage=rng.choice(["f32", "f32", "f32", "f32", "bf16", "f16_linear"]),
                        clip=data == "uniform" and mode == "composite" and rng.random() < 0.5)
        if more["storage"] == "f16_linear":
            nx, more["interp"] = (nx + 7) // 8 * 8, "trilinear"
        return _render("", nx, ny, nz, width, height, mode, **more)
    if kind == "maps":
        n = _logint(rng, 48, 700)
        return dict(kind="maps", nx=n, ny=n, nz=_logint(rng, 32, 900), width=rng.choice([n, 2 * n]), step=0.5,
                    **NOISE) | {"height": 0}
    if kind == "smooth":
        radius = rng.choice([1, 2, 3, 4, 6, 6, 8])
        nx, ny, nz = (_logint(rng, 40, 600) for _ in range(3))
        if rng.random() < 0.6:
            nx = (nx + 3) // 4 * 4
        return dict(kind="smooth", nx=nx, ny=ny, nz=nz, sigma=radius / 3.0, radius=radius, pair=rng.random() < 0.35)
    if kind == "batch":
        return dict(kind="batch", count=_logint(rng, 16, 400), lo_dim=32, hi_dim=_logint(rng, 64, 224),
                    size=rng.choice([96, 128, 200, 256]), layout=rng.randrange(1 << 20),
                    bricks=rng.choice(["none", "none", "half", "plan"]), step=0.5, opacity_scale=0.02, **NOISE)
    nx, ny, nz = (_logint(rng, 32, 256) for _ in range(3))
    return dict(kind="fit", nx=nx, ny=ny, nz=nz, width=_logint(rng, 64, 512), height=_logint(rng, 64, 512),
                yaw=round(rng.uniform(0, 360), 2), pitch=round(rng.uniform(-60, 60), 2), step=0.5,
                opacity_scale=rng.choice([0.02, 0.1]), ckpt_interval=64, **NOISE)


# ---- inputs ----------------------------------------------------------------------------------


def _lut():
    t = np.arange(256, dtype=np.float64) / 255.0
    return torch.from_numpy(np.stack([t, 1 - t, 0.5 + 0.5 * t, t], axis=1).astype(np.float32)).to(DEV)


def _frame(fwd):
    fwd = np.asarray(fwd, np.float64)
    fwd = fwd / np.linalg.norm(fwd)
    hint = np.array([0.0, 1.0, 0.0]) if abs(fwd[1]) <= 0.999 else np.array([0.0, 0.0, 1.0])
    right = np.cross(hint, fwd)
    right /= np.linalg.norm(right)
    return right, np.cross(fwd, right), fwd


def _camera(dims, yaw, pitch, width, height, ortho=False, fov=45.0):
    """A camera on the sphere that shows the whole cube, looking at its centre."""
    half = math.radians(fov) / 2
    radius = 0.5 * math.sqrt(sum(n * n for n in dims))
    y, p = math.radians(yaw), math.radians(pitch)
    right, up, fwd = _frame([math.sin(y) * math.cos(p), math.sin(p), math.cos(y) * math.cos(p)])
    eye = np.array([(n - 1) / 2 for n in dims]) - radius / math.sin(half) * fwd
    f = lambda v: np.asarray(v, np.float32)
    return SimpleNamespace(eye=f(eye), right=f(right), up=f(up), fwd=f(fwd),
                           tan_half_fovy=float(np.float32(math.tan(half))), ortho_half_h=float(np.float32(radius)),
                           ortho=bool(ortho), width=int(width), height=int(height))


def _axis_camera(dims, width, height):
    """Parallel rays down the spectral axis, the image covering the cube's face."""
    f = lambda v: np.asarray(v, np.float32)
    return SimpleNamespace(eye=f([(dims[0] - 1) / 2, (dims[1] - 1) / 2, -8.0]), right=f([1, 0, 0]), up=f([0, 1, 0]),
                           fwd=f([0, 0, 1]), tan_half_fovy=0.0, ortho_half_h=float(dims[1] / 2), ortho=True,
                           width=int(width), height=int(height))


def _dims(case):
    return case["nx"], case["ny"], case["nz"]


def _case_camera(case):
    if case["kind"] == "maps":
        n, w = case["nx"], case["width"]
        return _axis_camera(_dims(case), w, case["height"] or round(w * case["ny"] / n))
    if case.get("axis_view"):
        return _axis_camera(_dims(case), case["width"], case["height"])
    return _camera(_dims(case), case["yaw"], case["pitch"], case["width"], case["height"], case.get("ortho", False))


def _gen(seed, stream=0):
    return torch.Generator(device=DEV).manual_seed((seed * 1009 + stream * 7919 + 17) % (1 << 62))


def _add_sources(cube, rng, n, peak, sig, sig_z, margin=0.1):
    """Elliptical Gaussian sources whose centroid drifts along z with x, like a rotating disc."""
    nz, ny, nx = cube.shape
    for _ in range(n):
        smaj = math.exp(rng.uniform(math.log(sig[0]), math.log(sig[1])))
        smin, pa, grad = smaj * rng.uniform(0.4, 1.0), rng.uniform(0, math.pi), rng.uniform(-0.5, 0.5)
        cx, cy, cz = (rng.uniform(margin * m, (1 - margin) * m) for m in (nx, ny, nz))
        amp, ext = rng.uniform(*peak), 4 * smaj
        zext = 4 * sig_z + abs(grad) * ext
        x0, x1 = max(0, int(cx - ext)), min(nx, int(cx + ext) + 2)
        y0, y1 = max(0, int(cy - ext)), min(ny, int(cy + ext) + 2)
        z0, z1 = max(0, int(cz - zext)), min(nz, int(cz + zext) + 2)
        if x0 >= x1 or y0 >= y1 or z0 >= z1:
            continue
        x = torch.arange(x0, x1, device=DEV, dtype=torch.float32)[None, None, :] - cx
        y = torch.arange(y0, y1, device=DEV, dtype=torch.float32)[None, :, None] - cy
        z = torch.arange(z0, z1, device=DEV, dtype=torch.float32)[:, None, None] - cz
        c, s = math.cos(pa), math.sin(pa)
        plane = ((x * c + y * s) / smaj) ** 2 + ((y * c - x * s) / smin) ** 2
        cube[z0:z1, y0:y1, x0:x1] += amp * torch.exp(-0.5 * (plane + ((z - grad * x) / sig_z) ** 2))


def _cube(dims, data, seed, stream=0):
    nx, ny, nz = dims
    if data == "uniform":
        return torch.rand((nz, ny, nx), generator=_gen(seed, stream), device=DEV)
    cube = torch.randn((nz, ny, nx), generator=_gen(seed, stream), device=DEV)
    rng = random.Random(seed * 31 + stream)
    small = min(nx, ny)
    if data == "sources":
        _add_sources(cube, rng, max(3, min(200, nx * ny * nz // 1300000)), (2.0, 10.0),
                     (min(2.5, small / 12), min(17.0, small / 5)), 3.0)
    elif data == "stamp":
        _add_sources(cube, rng, 1, (5.0, 5.0), (small / 16, small / 8), max(1.0, 3.0 * nz / 64), margin=0.25)
    else:  # the mosaic: bright discs, and NaN outside a tilted square footprint
        _add_sources(cube, rng, 2, (30.0, 40.0), (small / 20, small / 12), nz / 10, margin=0.3)
        _add_sources(cube, rng, 30, (2.0, 10.0), (2.5, 12.0), 3.0, margin=0.2)
        y = torch.arange(ny, device=DEV, dtype=torch.float32)[:, None] - ny / 2
        x = torch.arange(nx, device=DEV, dtype=torch.float32)[None, :] - nx / 2
        c, s = math.cos(math.radians(30)), math.sin(math.radians(30))
        out = ((x * c + y * s).abs() > 0.36 * nx) | ((y * c - x * s).abs() > 0.36 * ny)
        cube.masked_fill_(out[None], float("nan"))
    return cube


def _second_line(first, seed):
    return first * 0.3 + torch.randn(first.shape, generator=_gen(seed, 5), device=DEV)


def _taps(case):
    """The N-tap binomial filter folded for linear sampling: centre weight, offsets, weights.
    The 9-tap one is the paper's, the central part of the 12-fold binomial."""
    n, drop = case["smooth_size"], 2 if case["smooth_size"] == 9 else 0
    w = np.array([math.comb(n - 1 + 2 * drop, k) for k in range(drop, n + drop)], np.float64)
    w /= w.sum()
    r, offs, wts = (n - 1) // 2, [], []
    for a in range(1, r + 1, 2):
        pair = [(k, w[r + k]) for k in (a, a + 1) if k <= r]
        s = sum(v for _, v in pair)
        offs.append(sum(k * v for k, v in pair) / s)
        wts.append(s)
    return float(w[r]), offs, wts


def _batch_layout(case):
    rng = random.Random(case["layout"])
    lo, hi = case["lo_dim"], case["hi_dim"]
    out = []
    for i in range(case["count"]):
        dims = tuple(min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))) for _ in range(3))
        cam = _camera(dims, rng.uniform(0, 360), rng.uniform(-60, 60), case["size"], case["size"])
        out.append((dims, cam, ("mip", "composite")[(i // 2) % 2], case["bricks"] == "half" and i % 2 == 1))
    return out


def _render_kwargs(case):
    kw = dict(interp=case["interp"], step=case["step"], lo=case["lo"], hi=case["hi"],
              opacity_scale=case["opacity_scale"], ratio_floor=case.get("ratio_floor", 0.0))
    if case["clip"]:
        kw.update(filter="clip", min_threshold=0.9, max_threshold=1.0)
    if case["smooth"] == "box":
        kw.update(smooth="box", smooth_arm=(case["smooth_size"] - 1) // 2)
    elif case["smooth"] == "gauss":
        kw.update(smooth="taps", smooth_taps=_taps(case))
    kw.update({k: case["outputs"] == "all" for k in ("scalar", "index", "nsamples")})
    return kw


def _volumes(case, seed):
    """(the cube, the second cube or None) as float32, before any packing."""
    first = _cube(_dims(case), case["data"], seed)
    return first, (_second_line(first, seed) if case["mode"] == "ratio" else None)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "smooth":
        cube = _cube(_dims(case), "sources", seed)
        st = dict(cube=cube, first=torch.randn(cube.shape, generator=_gen(seed, 5), device=DEV) if case["pair"] else None)
        st["out"] = torch.empty(tuple(cube.shape) + ((2,) if case["pair"] else ()), device=DEV)
        return dict(case=case, **st)
    if kind == "batch":
        # the stamps are drawn into one array of images
        images = torch.empty((case["count"], case["size"], case["size"], 4), dtype=torch.float32, device=DEV)
        items = []
        for i, (dims, cam, mode, brick) in enumerate(_batch_layout(case)):
            cube = _cube(dims, "stamp", seed, 100 + i)
            items.append((shw.pack_bricks(cube, "bf16") if brick else cube, cam, mode, images[i]))
        plan = shw.BatchPlan(items, lut=_lut(), step=case["step"], lo=case["lo"], hi=case["hi"],
                             opacity_scale=case["opacity_scale"], pack="bf16" if case["bricks"] == "plan" else None)
        return dict(case=case, plan=plan, images=images)
    cam, lut = _case_camera(case), _lut()
    if kind == "fit":
        cube = _cube(_dims(case), "stamp", seed).requires_grad_()
        target = torch.rand((cam.height, cam.width, 4), generator=_gen(seed, 9), device=DEV) * 0.6
        noisy = (lut + 0.05 * torch.randn(lut.shape, generator=_gen(seed, 10), device=DEV)).clamp(0, 1)
        return dict(case=case, cam=cam, cube=cube, lut=noisy.requires_grad_(), target=target,
                    scale=torch.tensor(case["opacity_scale"], device=DEV, requires_grad=True))
    if kind == "maps":
        return dict(case=case, cam=cam, lut=lut, cube=_cube(_dims(case), "sources", seed))
    first, second = _volumes(case, seed)
    st = dict(case=case, cam=cam, lut=lut, vol=first, vol2=None, kw=_render_kwargs(case))
    if case["mode"] == "ratio" and case["storage"] != "two":
        st["vol"] = torch.stack([first, second], dim=-1).contiguous()
    elif case["mode"] == "ratio":
        st["vol2"] = second
    # an interactive program draws into the same image every frame
    st["out"] = None if case["outputs"] == "all" else {
        "rgba": torch.empty((case["height"], case["width"], 4), dtype=torch.float32, device=DEV)}
    return st


# ---- one pass --------------------------------------------------------------------------------


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "smooth":
        if case["pair"]:
            return shw.smooth_zip(state["cube"], state["first"], case["sigma"], case["radius"], out=state["out"])
        return shw.smooth(state["cube"], case["sigma"], case["radius"], out=state["out"])
    if kind == "batch":
        state["plan"].render()
        return state["images"]
    if kind == "fit":
        img = shw.composite_render(state["cube"], state["lut"], state["scale"], state["cam"], step=case["step"],
                                   lo=case["lo"], hi=case["hi"], ckpt_interval=case["ckpt_interval"])
        loss = ((img - state["target"]) ** 2).mean()
        g_cube, g_lut, g_scale = torch.autograd.grad(loss, [state["cube"], state["lut"], state["scale"]])
        return {"rgba": img.detach(), "cube": g_cube, "lut": g_lut, "scale": g_scale}
    if kind == "maps":
        return [shw.render(state["cube"], state["cam"], mode, lut=state["lut"], step=case["step"], lo=case["lo"],
                           hi=case["hi"]) for mode in ("mip", "moment1")]
    vol, packed = state["vol"], None
    if case["storage"] in ("bf16", "f16_linear"):
        # the cube of this pass is new: it is packed, then its first view is drawn
        vol = shw.pack_bricks(vol, case["storage"])
        packed = vol.data
    out = shw.render(vol, state["cam"], case["mode"], lut=state["lut"], vol2=state["vol2"], out=state["out"],
                     **state["kw"])
    return out if packed is None else {**out, "packed": packed}


# ---- the work of one pass --------------------------------------------------------------------


def _count_samples(dims, cam, step):
    o, d = _rays(cam, "cpu")
    _, n = _clip(dims, o, d, float(np.float32(step)))
    return int(n.sum())


MODE_FLOPS = {"mip": 1, "avg": 1, "spectral": 1, "moment1": 6, "composite": 21, "ratio": 2}


def work(case):
    kind = case["kind"]
    if kind == "smooth":
        v = math.prod(_dims(case))
        return {"bytes": v * (16 if case["pair"] else 8), "flops": v * 6 * (2 * case["radius"] + 1)}
    if kind == "batch":
        b = f = 0
        for dims, cam, mode, brick in _batch_layout(case):
            n = _count_samples(dims, cam, case["step"])
            b += math.prod(dims) * (2 if brick or case["bricks"] == "plan" else 4) + case["size"] ** 2 * 16
            f += n * (24 + MODE_FLOPS[mode])
        return {"bytes": b, "flops": f}
    v, cam = math.prod(_dims(case)), _case_camera(case)
    n, px = _count_samples(_dims(case), cam, case["step"]), cam.width * cam.height
    if kind == "fit":
        # the cube, its gradient, the image, the target; forward, and twice that for the reverse
        return {"bytes": v * 8 + px * 32, "flops": n * 3 * (24 + MODE_FLOPS["composite"])}
    if kind == "maps":
        return {"bytes": 2 * (v * 4 + px * 28), "flops": n * (2 * 24 + MODE_FLOPS["mip"] + MODE_FLOPS["moment1"])}
    cubes = 2 if case["mode"] == "ratio" else 1
    fetches = 1
    if case["smooth"] == "box":
        fetches = case["smooth_size"]
    elif case["smooth"] == "gauss":
        fetches = 1 + 6 * len(_taps(case)[1])
    per_fetch = 24 if case["interp"] == "trilinear" else 0
    per_voxel = {"f32": 4, "two": 4, "pair": 4, "bf16": 6, "f16_linear": 6}[case["storage"]]
    return {"bytes": v * per_voxel * cubes + px * (28 if case["outputs"] == "all" else 16),
            "flops": n * (cubes * fetches * per_fetch + MODE_FLOPS[case["mode"]])}


# ---- the same in 64 bits ---------------------------------------------------------------------


def _f32(x):
    return float(np.float32(x))


def _rays(cam, dev):
    """Ray origins and unit directions, [3] lists of float64 vectors over the pixels."""
    w, h = cam.width, cam.height
    xs = (2.0 * (torch.arange(w, dtype=torch.float64, device=dev) + 0.5) / w - 1.0)[None, :].expand(h, w).reshape(-1)
    ys = (1.0 - 2.0 * (torch.arange(h, dtype=torch.float64, device=dev) + 0.5) / h)[:, None].expand(h, w).reshape(-1)
    eye, right, up, fwd = ([float(x) for x in getattr(cam, k)] for k in ("eye", "right", "up", "fwd"))
    aspect = w / h
    if cam.ortho:
        hh = _f32(cam.ortho_half_h)
        nf = math.sqrt(sum(x * x for x in fwd))
        o = [eye[a] + xs * (hh * aspect) * right[a] + ys * hh * up[a] for a in range(3)]
        return o, [torch.full_like(xs, fwd[a] / nf) for a in range(3)]
    t = _f32(cam.tan_half_fovy)
    u = [fwd[a] + xs * (t * aspect) * right[a] + ys * t * up[a] for a in range(3)]
    nu = torch.sqrt(u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
    return [torch.full_like(xs, eye[a]) for a in range(3)], [x / nu for x in u]


def _clip(dims, o, d, step):
    """The ray parameter at the box and the number of samples of each ray."""
    tmin, tmax = torch.full_like(o[0], -math.inf), torch.full_like(o[0], math.inf)
    miss = torch.zeros_like(o[0], dtype=torch.bool)
    for a in range(3):
        lo, hi, zero = -0.5, dims[a] - 0.5, d[a] == 0
        da = torch.where(zero, torch.ones_like(d[a]), d[a])
        ta, tb = (lo - o[a]) / da, (hi - o[a]) / da
        tmin = torch.where(zero, tmin, torch.maximum(tmin, torch.minimum(ta, tb)))
        tmax = torch.where(zero, tmax, torch.minimum(tmax, torch.maximum(ta, tb)))
        miss |= zero & ((o[a] < lo) | (o[a] > hi))
    t0 = tmin.clamp_min(0)
    n = torch.where(miss | ~(tmax > t0), torch.zeros_like(t0), torch.floor((tmax - t0) / step))
    return t0, n.long()


def _fetch(vol, dims, p, interp):
    flat = vol.reshape(-1)
    if interp == "nearest":
        i = [torch.floor(p[a] + 0.5).clamp_(0, dims[a] - 1).long() for a in range(3)]
        return flat[(i[2] * dims[1] + i[1]) * dims[0] + i[0]].double()
    lo, hi, f = [], [], []
    for a in range(3):
        fl = torch.floor(p[a])
        f.append(p[a] - fl)
        i = fl.long()
        stride = (1, dims[0], dims[0] * dims[1])[a]
        lo.append(i.clamp(0, dims[a] - 1) * stride)
        hi.append((i + 1).clamp_(0, dims[a] - 1) * stride)
    acc = None
    for cz in (lo, hi):
        wz = f[2] if cz is hi else 1 - f[2]
        for cy in (lo, hi):
            wzy = wz * (f[1] if cy is hi else 1 - f[1])
            base = cz[2] + cy[1]
            v = wzy * ((1 - f[0]) * flat[base + lo[0]].double() + f[0] * flat[base + hi[0]].double())
            acc = v if acc is None else acc + v
    return acc


def _lut_at(lut, vhat):
    u = 255.0 * vhat
    i = torch.floor(u).clamp_(0, 254)
    f = (u - i)[:, None]
    i = i.long()
    return (1 - f) * lut[i] + f * lut[i + 1]


def _norm(v, lo, hi):
    return ((v - lo) / (hi - lo)).clamp(0, 1)


def _march(case, vol, vol2, cam, lut, mode, chunk=1 << 20):
    """One render in 64 bits: (rgba, scalar) of every pixel."""
    dims = (vol.shape[2], vol.shape[1], vol.shape[0])
    step, lo, hi = _f32(case["step"]), _f32(case["lo"]), _f32(case["hi"])
    s, floor_ = _f32(case.get("opacity_scale", 1.0)), _f32(case.get("ratio_floor", 0.0))
    interp, smooth = case.get("interp", "trilinear"), case.get("smooth", "none")
    o_all, d_all = _rays(cam, DEV)
    t_all, n_all = _clip(dims, o_all, d_all, step)
    rgba = torch.zeros((cam.width * cam.height, 4), dtype=torch.float64, device=DEV)
    scalar = torch.zeros(cam.width * cam.height, dtype=torch.float64, device=DEV)
    c0, offs, wts = _taps(case) if smooth == "gauss" else (1.0, [], [])
    c0, offs, wts = _f32(c0), [_f32(x) for x in offs], [_f32(x) for x in wts]
    lut = lut.double()

    def value(cube, p, d):
        v = _fetch(cube, dims, p, interp)
        if smooth == "box":
            arm = (case["smooth_size"] - 1) // 2
            for i in range(1, arm + 1):
                for sign in (i, -i):
                    v = v + _fetch(cube, dims, [p[a] + sign * d[a] for a in range(3)], interp)
            v = v / (2 * arm + 1)
        elif smooth == "gauss":
            for axis in range(3):
                out = v * c0
                for off, w in zip(offs, wts):
                    for sign in (off, -off):
                        out = out + w * _fetch(cube, dims, [p[a] + sign if a == axis else p[a] for a in range(3)], interp)
                v = out
        return v

    order = torch.argsort(n_all, descending=True)
    order = order[: int((n_all > 0).sum())]
    for first in range(0, len(order), chunk):
        ids = order[first:first + chunk]
        n = n_all[ids]
        top = int(n[0])
        # rays still marching at sample k are a prefix: they are sorted by their counts
        alive_at = torch.searchsorted(-n.contiguous(), -torch.arange(top, device=DEV), right=False).tolist()
        o, d, t0 = [x[ids] for x in o_all], [x[ids] for x in d_all], t_all[ids]
        m = torch.full_like(t0, -math.inf)
        zmax, total, sw, szw = (torch.zeros_like(t0) for _ in range(4))
        trans, done = torch.ones_like(t0), torch.zeros_like(t0, dtype=torch.bool)
        col = torch.zeros((len(ids), 3), dtype=torch.float64, device=DEV)
        for k in range(top):
            r = slice(0, alive_at[k])
            t = t0[r] + (k + 0.5) * step
            dk = [x[r] for x in d]
            p = [o[a][r] + t * dk[a] for a in range(3)]
            v = value(vol, p, dk)
            if mode == "ratio":
                v = torch.where(v > floor_, value(vol2, p, dk) / v, torch.full_like(v, lo))
            v = torch.where(torch.isnan(v), torch.full_like(v, lo), v)
            if case.get("clip"):
                v = torch.where((v < _f32(0.9)) | (v > 1.0), torch.full_like(v, lo), v)
            z = p[2] if interp == "trilinear" else torch.floor(p[2] + 0.5).clamp(0, dims[2] - 1)
            if mode in ("mip", "ratio", "spectral"):
                new = v >= m[r]
                m[r] = torch.where(new, v, m[r])
                zmax[r] = torch.where(new, z, zmax[r])
            elif mode == "avg":
                total[r] += v
            elif mode == "moment1":
                w = (v - lo).clamp_min(0)
                total[r] += v
                sw[r] += w
                szw[r] += z * w
            else:
                c = _lut_at(lut, _norm(v, lo, hi))
                a = torch.where(done[r], torch.zeros_like(v), (s * c[:, 3]).clamp(0, 1))
                col[r] += (trans[r] * a)[:, None] * c[:, :3]
                trans[r] *= 1 - a
                done[r] |= (1 - trans[r]) > _f32(0.99)
        if mode in ("mip", "ratio"):
            sc, img = m, _lut_at(lut, _norm(m, lo, hi))
        elif mode == "avg":
            sc = total / n
            img = _lut_at(lut, _norm(sc, lo, hi))
        elif mode == "spectral":
            sc = m
            img = torch.cat([_lut_at(lut, ((zmax + 0.5) / dims[2]).clamp(0, 1))[:, :3], _norm(m, lo, hi)[:, None]], 1)
        elif mode == "moment1":
            some = sw > 0
            sc = torch.where(some, szw / sw, torch.zeros_like(sw))
            img = torch.cat([_lut_at(lut, ((sc + 0.5) / dims[2]).clamp(0, 1))[:, :3],
                             _norm(total / n, lo, hi)[:, None]], 1) * some[:, None]
        else:
            sc, img = 1 - trans, torch.cat([col, (1 - trans)[:, None]], 1)
        rgba[ids], scalar[ids] = img, sc
    return rgba.reshape(cam.height, cam.width, 4), scalar.reshape(cam.height, cam.width)


def _smooth64(cube, sigma, radius):
    k = torch.arange(-radius, radius + 1, dtype=torch.float64)
    w = torch.exp(-0.5 * (k / sigma) ** 2)
    w = (w / w.sum()).tolist()
    v = cube.double()
    for axis in range(3):
        n = v.shape[axis]
        out = torch.zeros_like(v)
        for j in range(-radius, radius + 1):
            i = (torch.arange(n, device=DEV) + j).clamp_(0, n - 1)
            out.add_(v.index_select(axis, i), alpha=w[j + radius])
        v = out
    return v


def _fit64(case, st):
    """The loss gradient of the compositing render, by the recurrences of its definition."""
    cube, lut, cam = st["cube"].detach(), st["lut"].detach().double(), st["cam"]
    s, lo, hi = _f32(case["opacity_scale"]), _f32(case["lo"]), _f32(case["hi"])
    dims, step = _dims(case), _f32(case["step"])
    o, d = _rays(cam, DEV)
    t0, n = _clip(dims, o, d, step)
    trans, col = torch.ones_like(t0), torch.zeros((len(t0), 3), dtype=torch.float64, device=DEV)
    done, tape = torch.zeros_like(t0, dtype=torch.bool), []
    for k in range(int(n.max())):
        ids = torch.nonzero((n > k) & ~done).squeeze(1)
        if not len(ids):
            break
        t = t0[ids] + (k + 0.5) * step
        v = _fetch(cube, dims, [o[a][ids] + t * d[a][ids] for a in range(3)], "trilinear")
        c = _lut_at(lut, _norm(v, lo, hi))
        a = (s * c[:, 3]).clamp(0, 1)
        tape.append((k, ids, v, trans[ids]))
        col[ids] += (trans[ids] * a)[:, None] * c[:, :3]
        trans[ids] *= 1 - a
        done[ids] = (1 - trans[ids]) > _f32(0.99)
    img = torch.cat([col, (1 - trans)[:, None]], 1)
    g = 2.0 * (img - st["target"].double().reshape(-1, 4)) / img.numel()
    g_cube = torch.zeros(math.prod(dims), dtype=torch.float64, device=DEV)
    g_lut = torch.zeros_like(lut)
    g_scale = torch.zeros((), dtype=torch.float64, device=DEV)
    below = -g[:, 3].clone()  # the loss per unit of transmittance reaching the samples behind
    for k, ids, v, tk in reversed(tape):
        x = (v - lo) / (hi - lo)
        vh = x.clamp(0, 1)
        c = _lut_at(lut, vh)
        raw = s * c[:, 3]
        a = raw.clamp(0, 1)
        gc = (g[ids, :3] * c[:, :3]).sum(1)
        d_a = tk * (gc - below[ids])
        below[ids] = a * gc + (1 - a) * below[ids]
        d_raw = torch.where((raw >= 0) & (raw <= 1), d_a, torch.zeros_like(d_a))
        g_scale += (d_raw * c[:, 3]).sum()
        d_c = torch.cat([(tk * a)[:, None] * g[ids, :3], (s * d_raw)[:, None]], 1)
        u = 255.0 * vh
        i = torch.floor(u).clamp_(0, 254)
        f = (u - i)[:, None]
        i = i.long()
        g_lut.index_add_(0, i, (1 - f) * d_c)
        g_lut.index_add_(0, i + 1, f * d_c)
        slope = 255.0 / (hi - lo) * (d_c * (lut[i + 1] - lut[i])).sum(1)
        d_v = torch.where((x >= 0) & (x <= 1), slope, torch.zeros_like(slope))
        t = t0[ids] + (k + 0.5) * step
        lo_i, hi_i, fr = [], [], []
        for ax in range(3):
            p = o[ax][ids] + t * d[ax][ids]
            fl = torch.floor(p)
            fr.append(p - fl)
            stride = (1, dims[0], dims[0] * dims[1])[ax]
            lo_i.append(fl.long().clamp(0, dims[ax] - 1) * stride)
            hi_i.append((fl.long() + 1).clamp(0, dims[ax] - 1) * stride)
        for corner in range(8):
            idx, w = 0, d_v
            for ax in range(3):
                up = corner >> ax & 1
                idx = idx + (hi_i[ax] if up else lo_i[ax])
                w = w * (fr[ax] if up else 1 - fr[ax])
            g_cube.index_add_(0, idx, w)
    return {"rgba": img.reshape(cam.height, cam.width, 4), "cube": g_cube.reshape(cube.shape), "lut": g_lut,
            "scale": g_scale}


def exact(case, seed):
    kind = case["kind"]
    if kind == "smooth":
        cube = _cube(_dims(case), "sources", seed)
        out = _smooth64(cube, _f32(case["sigma"]), case["radius"])
        if not case["pair"]:
            return out
        first = torch.randn(cube.shape, generator=_gen(seed, 5), device=DEV)
        return torch.stack([first.double(), out], dim=-1)
    if kind == "batch":
        if case["count"] > 60:  # thousands of short marches: too slow in plain torch
            return None
        lut, out = _lut(), []
        for i, (dims, cam, mode, brick) in enumerate(_batch_layout(case)):
            cube = _cube(dims, "stamp", seed, 100 + i)
            if brick or case["bricks"] == "plan":
                cube = cube.bfloat16().float()
            out.append(_march(case, cube, None, cam, lut, mode)[0])
        return torch.stack(out)
    cam, lut = _case_camera(case), _lut()
    if kind == "fit":
        return _fit64(case, prepare(case, seed))
    if kind == "maps":
        cube = _cube(_dims(case), "sources", seed)
        out = []
        for mode in ("mip", "moment1"):
            rgba, scalar = _march(case, cube, None, cam, lut, mode)
            out.append({"rgba": rgba, "scalar": scalar, "index": None, "nsamples": None})
        return out
    first, second = _volumes(case, seed)
    packed = case["storage"] in ("bf16", "f16_linear")
    if packed:
        half = torch.bfloat16 if case["storage"] == "bf16" else torch.float16
        first, second = (v if v is None else v.to(half).float() for v in (first, second))
    rgba, scalar = _march(case, first, second, cam, lut, case["mode"])
    out = {"rgba": rgba}
    if case["outputs"] == "all":
        out.update(scalar=scalar, index=None, nsamples=None)
    if packed:
        out["packed"] = None
    return out
