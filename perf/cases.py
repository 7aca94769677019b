"""The workloads the library's speed is measured on, each one pass of work that a
user's program has the public API do.

A case names a kind of work and its sizes:

  view       a rendered frame through geer.Renderer.forward (the pair count is
             checked on the host, as an interactive viewer does)
  stream     a rendered frame through geer.Workspace without a host check (an
             offline or streaming renderer)
  noalloc    one small frame through geer_render_noalloc (embedded renderers)
  serve      a batch of camera requests of mixed models and sizes on one resident
             scene, through fixed camera slots (the serving loop's step)
  train      a training step: preprocess, binning, fused forward + L1 + backward,
             gradients of every parameter written
  autograd   the same step through the differentiable geer.render and a torch loss
  optimise   one Adam step over all Gaussian parameters
  refine     one density-control pass (classify, clone, split, prune, moments)
  evaluate   a finished render's evaluation: supervision image from the native
             camera, reprojection to the native image, regions, PSNR / SSIM

Scenes follow the distributions of paper_2505_24053_gb300.workloads (a cube in
front of the camera, a shell around it, a slab, a room of wall surfels), drawn on
the GPU from the seed.
"""
import copy
import ctypes
import math

import numpy as np
import torch

from paper_2505_24053_gb300 import geer
from paper_2505_24053_gb300 import workloads as wl

MODELS = {"pinhole": wl.PINHOLE, "equidistant": wl.EQUIDISTANT, "kb": wl.KANNALA_BRANDT}
NAMES = ("mean", "scale", "quat", "opacity", "sh")


def listed():
    return [
        # the smallest frame: workload 1, what a viewer redraws on every mouse move; latency and launches
        dict(name="view_small", kind="view", scene="cube", n=4096, deg=0, model="pinhole", w=128, h=128, fov=60.0),
        # an embedded renderer's small fisheye frame without any allocation
        dict(name="noalloc_small", kind="noalloc", scene="cube", n=12001, deg=1, model="kb", w=317, h=243, fov=150.0),
        # the gradient-check size (a 2048-Gaussian subset of workload 3 at 64 x 64): a first fit, a unit-sized step
        dict(name="autograd_small", kind="autograd", scene="cube", n=2048, deg=3, model="kb", w=64, h=64, fov=190.0),
        # an ordinary half-sphere frame of small, far Gaussians (workload 2)
        dict(name="stream_fisheye", kind="stream", scene="shell", n=500_000, deg=3, model="equidistant", w=1024,
             h=1024, fov=180.0),
        # the benchmark's training step (workload 3): 1M Gaussians, 190 degree Kannala-Brandt fisheye
        dict(name="train_fisheye", kind="train", scene="cube", n=1_000_000, deg=3, model="kb", w=1280, h=960,
             fov=190.0, cams=1, splat=False),
        # an indoor scene trained through autograd, ragged sizes, degree 2
        dict(name="autograd_room", kind="autograd", scene="room", n=300_001, deg=2, model="equidistant", w=801, h=599,
             fov=170.0),
        # one batch of the serving mix (workload 4) on its 2M-Gaussian scene
        dict(name="serve_mix", kind="serve", scene="cube", n=2_000_000, deg=3, requests=3),
        # the large scene (workload 5): four surround cameras in one launch, forward and backward
        dict(name="train_surround", kind="train", scene="slab", n=6_000_000, deg=3, model="equidistant", w=1920,
             h=1536, fov=210.0, cams=4, splat=False),
        # training with the local-affine splat alpha and its EWA association (the ablation's training variant)
        dict(name="train_splat", kind="train", scene="cube", n=250_000, deg=1, model="pinhole", w=960, h=720,
             fov=90.0, cams=1, splat=True),
        # the optimiser after some refinements: counts are whatever density control left
        dict(name="optimise", kind="optimise", n=1_093_217, deg=3),
        # density control of the 1M-Gaussian scene, about 9% densified
        dict(name="refine", kind="refine", n=1_000_000, deg=3),
        # evaluation of one native fisheye image
        dict(name="evaluate", kind="evaluate", model="kb", w=1280, h=960, fov=190.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["view", "stream", "noalloc", "serve", "train", "train", "autograd", "optimise", "refine",
                       "evaluate"])
    deg = rng.randint(0, 3)
    if kind in ("optimise", "refine"):
        return dict(kind=kind, n=_log(rng, 20_000, 2_000_000), deg=deg)
    model = rng.choice(["pinhole", "equidistant", "kb"])
    fov = round(rng.uniform(55, 110) if model == "pinhole" else rng.uniform(120, 210 if model == "equidistant" else 190), 2)
    if kind == "evaluate":
        w = _log(rng, 200, 1920)
        return dict(kind=kind, model=model, w=w, h=int(w * rng.uniform(0.5, 0.95)), fov=fov)
    if kind == "serve":
        return dict(kind=kind, scene="cube", n=_log(rng, 50_000, 2_000_000), deg=deg, requests=rng.randint(1, 4))
    if kind == "noalloc":
        w = _log(rng, 48, 500)
        return dict(kind=kind, scene=rng.choice(["cube", "shell"]), n=_log(rng, 200, 30_000), deg=deg, model=model,
                    w=w, h=int(w * rng.uniform(0.5, 1.0)), fov=fov)
    scene = rng.choice(["cube", "cube", "shell", "room", "slab"])
    w = _log(rng, 60, 1900)
    big = kind in ("stream", "train")
    c = dict(kind=kind, scene=scene, n=_log(rng, 1500, 2_000_000 if big else 500_000), deg=deg, model=model,
             w=w, h=int(min(1500, w * rng.uniform(0.5, 1.0))), fov=fov)
    if kind == "train":
        c["cams"] = rng.choice([1, 1, 1, 2])
        c["splat"] = rng.random() < 0.2
    return c


# ---- inputs ---------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _uni(g, shape, lo, hi):
    return torch.rand(shape, generator=g, device="cuda") * (hi - lo) + lo


def _nrm(g, shape, mu, sd):
    return torch.randn(shape, generator=g, device="cuda") * sd + mu


def _quats(g, n):
    q = torch.randn((n, 4), generator=g, device="cuda")
    return q / q.norm(dim=1, keepdim=True)


def _params(case, g):
    """(mean, log_scale, quat, logit opacity, sh) of the case's scene."""
    n, deg, kind = case["n"], case["deg"], case.get("scene", "cube")
    if kind == "cube":
        mean = torch.cat([_uni(g, (n, 2), -2, 2), _uni(g, (n, 1), 3, 7)], 1)
        log_s, logit = _nrm(g, (n, 3), -2.5, 0.5), _nrm(g, (n,), 0.0, 1.0)
    elif kind == "shell":
        v = torch.randn((n, 3), generator=g, device="cuda")
        mean = v / v.norm(dim=1, keepdim=True) * _uni(g, (n, 1), 18, 22)
        log_s, logit = _nrm(g, (n, 3), -4.0, 0.7), _nrm(g, (n,), 0.0, 1.5)
    elif kind == "slab":
        mean = _uni(g, (n, 3), -1, 1) * torch.tensor([50.0, 5.0, 50.0], device="cuda")
        log_s, logit = _nrm(g, (n, 3), -3.5, 1.0), _nrm(g, (n,), 0.0, 1.0)
    else:  # room: 80% of the Gaussians flat on the walls (thin along the wall's axis), 20% clutter inside
        half = torch.tensor([2.5, 1.4, 3.0], device="cuda")
        ns = int(round(0.8 * n))
        area = torch.stack([half[1] * half[2], half[0] * half[2], half[0] * half[1]])
        ax = torch.multinomial(area, ns, replacement=True, generator=g)
        sign = torch.where(torch.rand(ns, generator=g, device="cuda") < 0.5, -1.0, 1.0)
        ms = _uni(g, (ns, 3), -1, 1) * half
        ms[torch.arange(ns, device="cuda"), ax] = sign * half[ax] + _nrm(g, (ns,), 0.0, 0.01)
        ls = _nrm(g, (ns, 3), -3.0, 0.8)
        ls[torch.arange(ns, device="cuda"), ax] = _nrm(g, (ns,), -5.5, 0.5)
        qs = torch.cat([torch.ones((ns, 1), device="cuda"), _nrm(g, (ns, 3), 0.0, 0.075)], 1)
        mean = torch.cat([ms, _uni(g, (n - ns, 3), -0.7, 0.7) * half])
        log_s = torch.cat([ls, _nrm(g, (n - ns, 3), -3.0, 0.7)])
        quat = torch.cat([qs / qs.norm(dim=1, keepdim=True), _quats(g, n - ns)])
        logit = _nrm(g, (n,), 1.0, 1.5)
    if kind != "room":
        quat = _quats(g, n)
    k = (deg + 1) ** 2
    sh = _nrm(g, (n, k, 3), 0.0, 0.2)
    sh[:, 0, :] = _uni(g, (n, 3), -math.sqrt(math.pi), math.sqrt(math.pi))
    return mean.contiguous(), log_s, quat, logit, sh.contiguous()


def _gaussians(case, g):
    mean, log_s, quat, logit, sh = _params(case, g)
    return geer.Gaussians(mean, torch.exp(log_s), quat, torch.sigmoid(logit), sh, case["deg"])


def _camera(case, yaw=0.0):
    R, t = wl.pose(wl.rot_y(math.radians(yaw)), (0, 0, 0))
    k = wl.kb_coeffs(3) if case["model"] == "kb" else (0.0, 0.0, 0.0, 0.0)
    return wl.Camera(MODELS[case["model"]], case["w"], case["h"], math.radians(case["fov"]), k=k, R_cw=R, t_cw=t)


def _cameras(case):
    n = case.get("cams", 1)
    return [_camera(case, 360.0 * i / n) for i in range(n)]


def _image(g, h, w):
    """A smooth image in [0, 1] with a little noise."""
    j, i = torch.meshgrid(torch.arange(h, device="cuda") / h, torch.arange(w, device="cuda") / w, indexing="ij")
    f, p = _uni(g, (3, 2), 1, 4), _uni(g, (3, 2), 0, 2 * math.pi)
    img = torch.stack([0.5 + 0.25 * torch.sin(2 * math.pi * f[c, 0] * i + p[c, 0])
                       + 0.2 * torch.cos(2 * math.pi * f[c, 1] * j + p[c, 1]) for c in range(3)], -1)
    return (img + _uni(g, (h, w, 3), -0.05, 0.05)).clamp(0, 1).contiguous()


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    s = {"case": case}
    if kind == "optimise":
        s["adam"] = geer.Adam(*_params(case, g), case["deg"], lr_mean=1e-3)
        raw = s["adam"].raw
        s["grads"] = {k: _nrm(g, raw[r].shape, 0.0, 1e-5) for k, r in
                      zip(NAMES, ("mean", "log_scale", "quat", "logit_opacity", "sh"))}
        s["adam"].m.copy_(_nrm(g, s["adam"].m.shape, 0.0, 1e-5))
        s["adam"].v.copy_(_uni(g, s["adam"].v.shape, 0.2, 2.0) * 1e-10)
        s["adam"].t = 500
        return s
    if kind == "refine":
        n = case["n"]
        mean, log_s, quat, logit, sh = _params(case, g)
        # a refinement's mix in fixed shares: 1% pruned (faint), 9% densified (their mean gradient above the
        # threshold; split or cloned by their size), the rest kept
        at = torch.randperm(n, generator=g, device="cuda")
        logit = logit.clamp(min=-5.0)
        logit[at[:n // 100]] = -6.0
        grad = _uni(g, (n,), 0.0, 1.9e-4)
        grad[at[n // 100:n // 10]] += 2.5e-4
        s["adam"] = geer.Adam(mean, log_s, quat, logit, sh, case["deg"])
        s["adam"].m.copy_(_nrm(g, s["adam"].m.shape, 0.0, 1e-5))
        s["adam"].v.copy_(_uni(g, s["adam"].v.shape, 0.2, 2.0) * 1e-10)
        s["denom"] = torch.floor(_uni(g, (n,), 1, 100))
        s["accum"] = s["denom"] * grad
        s["z"] = torch.randn((n, 2, 3), generator=g, device="cuda")
        return s
    if kind == "evaluate":
        s["cam"] = _camera(case)
        s["beap"], s["gt"] = _image(g, case["h"], case["w"]), _image(g, case["h"], case["w"])
        s["gt"] = (0.8 * s["beap"] + 0.2 * s["gt"]).contiguous()  # a reference near the render
        return s
    s["g"] = _gaussians(case, g)
    if kind == "serve":
        rng = np.random.default_rng(seed)
        s["cams"] = []
        for i in range(case["requests"]):
            model, w, h, fov, kseed = wl.SERVING_KINDS[i % 3]
            R, t = wl.random_pose(rng)
            s["cams"].append(wl.Camera(model, w, h, math.radians(fov), R_cw=R, t_cw=t,
                                       k=wl.kb_coeffs(kseed) if kseed is not None else (0.0, 0.0, 0.0, 0.0)))
        m = case["requests"]
        s["slot_pixels"], s["slot_tiles"] = 1920 * 1280, 120 * 80
        cap = wl.Camera(wl.PINHOLE, 1920, 1280, math.radians(60))
        pairs = 1000 + 30 * m * case["n"]
        while True:  # a server calibrates its pair capacity on its requests
            s["ws"] = ws = geer.Workspace([cap] * m, case["n"], case["deg"], pairs)
            ws.set_camera_slots(s["cams"], [True] * m, s["slot_tiles"], s["slot_pixels"])
            ws.preprocess(s["g"])
            try:
                ws.bin_sort()
                break
            except geer.GeerError as e:
                if e.status != geer.ERR_CAPACITY:
                    raise
                pairs = int(1.25 * ws.last_pairs) + 1024
        s["rgb"] = torch.zeros((m * s["slot_pixels"], 3), device="cuda")
        return s
    cams = _cameras(case)
    pixels = sum(c.pixels for c in cams)
    if kind == "noalloc":
        s["cam"] = geer.camera_c(cams[0])
        s["gc"] = s["g"].c_struct()
        s["rgb"], s["T"] = torch.empty((pixels, 3), device="cuda"), torch.empty(pixels, device="cuda")
        return s
    params = geer.params_c(assoc=geer.ASSOC_EWA, snugbox=True, alpha_model=geer.ALPHA_SPLAT) if case.get("splat") else None
    s["r"] = geer.Renderer(cams, case["n"], case["deg"], params=params)
    s["target"] = _uni(g, (pixels, 3), 0, 1)
    s["rgb"] = torch.empty((pixels, 3), device="cuda")
    if kind != "view":
        s["r"].prepare(s["g"])  # sizes the pair capacity; a program's steps stay asynchronous after it
    if kind == "train":
        s["dL"], s["loss"] = torch.empty_like(s["rgb"]), torch.empty(1, device="cuda")
        s["grads"] = {k: torch.empty_like(getattr(s["g"], k)) for k in NAMES}
    if kind == "autograd":
        s["leaves"] = [getattr(s["g"], k).clone().requires_grad_(True) for k in NAMES]
    return s


# ---- one pass -------------------------------------------------------------

def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "view":
        return s["r"].forward(s["g"], rgb=s["rgb"])
    if kind == "stream":
        ws = s["r"].ws
        ws.preprocess(s["g"])
        ws.bin_sort(sync=False)
        ws.render_fwd(s["rgb"])
        return s["rgb"]
    if kind == "noalloc":
        p = ctypes.c_void_p
        st = geer.lib().geer_render_noalloc(ctypes.byref(s["gc"]), ctypes.byref(s["cam"]), None, p(s["rgb"].data_ptr()),
                                            p(s["T"].data_ptr()), p(torch.cuda.current_stream().cuda_stream))
        if st != geer.OK:
            raise geer.GeerError(st, "geer_render_noalloc")
        return [s["rgb"], s["T"]]
    if kind == "serve":
        ws = s["ws"]
        ws.set_camera_slots(s["cams"], [True] * len(s["cams"]), s["slot_tiles"], s["slot_pixels"])
        ws.preprocess(s["g"])
        ws.bin_sort(sync=False)
        ws.render_fwd(s["rgb"])
        return [s["rgb"][i * s["slot_pixels"]:i * s["slot_pixels"] + c.pixels] for i, c in enumerate(s["cams"])]
    if kind == "train":
        ws = s["r"].ws
        ws.preprocess(s["g"])
        ws.bin_sort(sync=False)
        ws.render_train_l1(s["target"], s["rgb"], s["dL"], s["loss"])
        ws.preprocess_bwd(s["g"], s["grads"], accumulate=False)
        return {"rgb": s["rgb"], "loss": s["loss"], **s["grads"]}
    if kind == "autograd":
        for t in s["leaves"]:
            t.grad = None
        rgb = geer.render(s["r"], *s["leaves"], case["deg"])
        loss = (rgb - s["target"]).abs().mean()
        loss.backward()
        return {"rgb": rgb.detach(), "loss": loss.detach(), **{k: t.grad for k, t in zip(NAMES, s["leaves"])}}
    if kind == "optimise":
        a = s["adam"]
        a.step(s["grads"])
        return {**a.raw, "m": a.m, "v": a.v, "scale": a.gaussians.scale, "opacity": a.gaussians.opacity}
    if kind == "refine":
        a = copy.copy(s["adam"])  # densify replaces the attributes, not the tensors: the state keeps its own
        n = a.densify(s["accum"], s["denom"], s["z"], clone_max_scale=0.12)
        return {**a.raw, "m": a.m, "v": a.v, "scale": a.gaussians.scale, "opacity": a.gaussians.opacity, "n": n}
    cam = s["cam"]
    sup, valid = geer.native_to_beap(s["gt"], cam)
    native = geer.remap_to_native(s["beap"], cam)
    regions = geer.native_regions(cam)
    met = geer.image_metrics(native, s["gt"], regions, 2)
    return {"supervision": sup, "valid": valid, "native": native, "regions": regions,
            "metrics": [[m["sse"], m["ssim_sum"], m["count"]] for m in met]}


# ---- the work a pass cannot do without -------------------------------------

# contributors composited per ray: the number a dense scene saturates at, and the Gaussians at which it does
# (measured on the listed scenes; the cube's at a 60 degree field of view, it fills less of a wider one)
_DENSE = {"cube": (30.0, 4096), "shell": (50.0, 15_000_000), "slab": (55.0, 3_000_000), "room": (52.0, 100_000)}


def work(case):
    kind, deg = case["kind"], case.get("deg", 0)
    per = 11 + 3 * (deg + 1) ** 2
    if kind == "optimise":
        return {"bytes": case["n"] * (28 * per + 16), "flops": case["n"] * per * 14}
    if kind == "refine":
        # parameters and both moments read per input, written per output (1.08 outputs per input)
        return {"bytes": case["n"] * (12 * per * 2.08 + 8 + 24 + 16 * 1.08), "flops": case["n"] * 40}
    if kind == "evaluate":
        p = case["w"] * case["h"]
        return {"bytes": p * (12 * 4 + 2 + 12), "flops": p * (120 + 150 + 3 * 22 * 10)}
    if kind == "serve":
        pix = sum(wl.SERVING_KINDS[i % 3][1] * wl.SERVING_KINDS[i % 3][2] for i in range(case["requests"]))
        items = case["n"] * case["requests"]
    else:
        pix = case["w"] * case["h"] * case.get("cams", 1)
        items = case["n"] * case.get("cams", 1)
    c, at = _DENSE[case["scene"]]
    if case["scene"] == "cube":
        at *= (case.get("fov", 120.0) / 60.0) ** 2
    hits = pix * c * min(1.0, case["n"] / at)
    back = kind in ("train", "autograd")
    # Gaussians and image; training: target read, gradients written
    return {"bytes": case["n"] * 4 * per * (2 if back else 1) + pix * 12 * (2 if back else 1),
            "flops": items * 600 * (2 if back else 1) + hits * (66 + (132 if back else 0))}


# ---- 64-bit values ----------------------------------------------------------

F64 = torch.float64


def _kb(k, p):
    p2 = p * p
    return p * (1 + p2 * (k[0] + p2 * (k[1] + p2 * (k[2] + p2 * k[3]))))


def _geometry(cam):
    """(fov_x, fov_y, focal, k) in 64 bits from the camera's 32-bit fields."""
    fx, k = float(np.float32(cam.fov_x)), [float(np.float32(v)) for v in cam.k]
    if cam.model == wl.PINHOLE:
        return fx, 2 * math.atan(math.tan(fx / 2) * cam.height / cam.width), 0.5 * cam.width / math.tan(fx / 2), k
    edge = _kb(k, fx / 2)
    target, lo, hi = edge * cam.height / cam.width, 0.0, fx / 2
    for i in range(1, 8193):  # the smallest angle that reaches the target
        if _kb(k, fx / 2 * i / 8192) >= target:
            lo, hi = fx / 2 * (i - 1) / 8192, fx / 2 * i / 8192
            break
    else:
        return fx, None, None, k
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        lo, hi = (lo, mid) if _kb(k, mid) >= target else (mid, hi)
    return fx, 2 * hi, 0.5 * cam.width / edge, k


def _angles(cam, fx, fy):
    i = torch.arange(cam.width, device="cuda", dtype=F64)
    j = torch.arange(cam.height, device="cuda", dtype=F64)
    return ((i + 0.5) / cam.width - 0.5) * fx, ((j + 0.5) / cam.height - 0.5) * fy


def _sh_basis(deg, d):
    x, y, z = d.unbind(1)
    Y = [torch.full_like(x, 0.5 / math.sqrt(math.pi))]
    if deg > 0:
        a = math.sqrt(3 / (4 * math.pi))
        Y += [-a * y, a * z, -a * x]
    if deg > 1:
        a = math.sqrt(15 / math.pi) / 2
        Y += [a * x * y, -a * y * z, math.sqrt(5 / math.pi) / 4 * (3 * z * z - 1), -a * x * z, a / 2 * (x * x - y * y)]
    if deg > 2:
        a, b, c = math.sqrt(35 / (2 * math.pi)) / 4, math.sqrt(105 / math.pi) / 2, math.sqrt(21 / (2 * math.pi)) / 4
        Y += [-a * y * (3 * x * x - y * y), b * x * y * z, -c * y * (5 * z * z - 1),
              math.sqrt(7 / math.pi) / 4 * z * (5 * z * z - 3), -c * x * (5 * z * z - 1), b / 2 * z * (x * x - y * y),
              -a * x * (x * x - 3 * y * y)]
    return torch.stack(Y, 1)


def _render64(cam, mean, scale, quat, opacity, sh, deg):
    """[h*w, 3] image and transmittance: every ray against every Gaussian (mean .. sh: 64-bit tensors)."""
    fx, fy, _, _ = _geometry(cam)
    f32 = lambda v: float(np.float32(v))  # noqa: E731
    amin, tmin, amax = f32(1 / 255), f32(1e-4), f32(0.99)
    R = torch.tensor(np.asarray(cam.R_cw, np.float64), device="cuda")
    t = torch.tensor(np.asarray(cam.t_cw, np.float64), device="cuda")
    q = quat / quat.norm(dim=1, keepdim=True)
    w, x, y, z = q.unbind(1)
    Rq = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                      2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                      2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    mc = mean @ R.T + t
    W = (R @ Rq).transpose(1, 2) / scale[:, :, None]
    ou = -(W @ mc[:, :, None])[:, :, 0]
    with torch.no_grad():
        live = (opacity >= amin) & ((ou * ou).sum(1) > 2 * torch.log(opacity / amin) * (1 + 1e-3))
        order = torch.argsort(mc.norm(dim=1), stable=True)
        order = order[live[order]]
    d = mean + R.T @ t
    d = d / d.norm(dim=1, keepdim=True)
    col = ((_sh_basis(deg, d)[:, :, None] * sh).sum(1) + 0.5).clamp(min=0)
    W, ou, col, op = W[order], ou[order], col[order], opacity[order]
    th, ph = _angles(cam, fx, fy)
    st, ct, sp, cp = th.sin(), th.cos(), ph.sin(), ph.cos()
    rays = torch.stack([st[None, :] * cp[:, None], ct[None, :] * sp[:, None], ct[None, :] * cp[:, None]], -1).view(-1, 3)
    bg = torch.tensor([f32(v) for v in cam.bg], dtype=F64, device="cuda")
    rgb, Ts = [], []
    step = max(1, (1 << 22) // max(1, order.numel()))
    for a in range(0, rays.shape[0], step):
        r = rays[a:a + step]
        du = [r @ W[:, k, :].T for k in range(3)]
        o = [ou[:, k][None, :] for k in range(3)]
        m = [o[1] * du[2] - o[2] * du[1], o[2] * du[0] - o[0] * du[2], o[0] * du[1] - o[1] * du[0]]
        kap = (m[0] ** 2 + m[1] ** 2 + m[2] ** 2) / (du[0] ** 2 + du[1] ** 2 + du[2] ** 2)
        raw = op[None, :] * torch.exp(-kap / 2)
        hit = (raw >= amin) & (o[0] * du[0] + o[1] * du[1] + o[2] * du[2] < 0)
        al = torch.where(hit, raw.clamp(max=amax), torch.zeros_like(raw))
        Tn = torch.cumprod(1 - al, 1)
        use = torch.cummax((hit & (Tn < tmin)).to(torch.int8), 1).values == 0
        al = torch.where(use, al, torch.zeros_like(al))
        Tn = torch.cumprod(1 - al, 1)
        T0 = torch.cat([torch.ones_like(Tn[:, :1]), Tn[:, :-1]], 1)
        T = Tn[:, -1:] if Tn.shape[1] else torch.ones((r.shape[0], 1), dtype=F64, device="cuda")
        rgb.append((al * T0) @ col + T * bg)
        Ts.append(T[:, 0])
    return torch.cat(rgb), torch.cat(Ts)


def _bilinear(img, u, v):
    h, w = img.shape[:2]
    u, v = u.clamp(0, w - 1), v.clamp(0, h - 1)
    x0, y0 = u.long().clamp(max=max(w - 2, 0)), v.long().clamp(max=max(h - 2, 0))
    x1, y1 = (x0 + 1).clamp(max=w - 1), (y0 + 1).clamp(max=h - 1)
    ax, ay = (u - x0)[..., None], (v - y0)[..., None]
    top = img[y0, x0] + ax * (img[y0, x1] - img[y0, x0])
    return top + ay * (img[y1, x0] + ax * (img[y1, x1] - img[y1, x0]) - top)


def _evaluate64(s):
    cam, gt, beap = s["cam"], s["gt"].to(F64), s["beap"].to(F64)
    w, h = cam.width, cam.height
    fx, fy, f, k = _geometry(cam)
    if fy is None:
        return None
    ps = torch.arange(1, 4097, dtype=F64) * (math.pi / 4096)
    val = _kb(k, ps)
    fall = torch.nonzero(val <= torch.cat([torch.zeros(1, dtype=F64), val[:-1]]))
    pmax = math.pi if not len(fall) else math.pi * int(fall[0]) / 4096
    # supervision: each BEAP ray projected into the native image
    th, ph = _angles(cam, fx, fy)
    st, ct, sp, cp = th.sin()[None, :], th.cos()[None, :], ph.sin()[:, None], ph.cos()[:, None]
    d = torch.stack([st * cp, ct * sp, ct * cp], -1)
    rho = d[..., :2].norm(dim=-1)
    if cam.model == wl.PINHOLE:
        ok = d[..., 2] > 0
        sc = f / d[..., 2]
    else:
        p = torch.atan2(rho, d[..., 2])
        ok = p <= pmax
        sc = torch.where(rho > 0, f * _kb(k, p) / rho.clamp(min=1e-300), torch.zeros_like(rho))
    u, v = sc * d[..., 0] + 0.5 * w - 0.5, sc * d[..., 1] + 0.5 * h - 0.5
    ok &= (u >= -0.5) & (u <= w - 0.5) & (v >= -0.5) & (v <= h - 0.5)
    z = torch.zeros((), dtype=F64, device="cuda")
    sup = torch.where(ok[..., None], _bilinear(gt, torch.where(ok, u, z), torch.where(ok, v, z)), z)
    # native image: each native pixel's ray, its BEAP angles, the render there
    i = (torch.arange(w, device="cuda", dtype=F64) + 0.5 - 0.5 * w) / f
    j = (torch.arange(h, device="cuda", dtype=F64) + 0.5 - 0.5 * h) / f
    uu, vv = i[None, :].expand(h, w), j[:, None].expand(h, w)
    if cam.model == wl.PINHOLE:
        dx, dy, dz = uu, vv, torch.ones_like(uu)
        inv = torch.ones_like(uu, dtype=torch.bool)
    else:
        rd = (uu * uu + vv * vv).sqrt()
        lo, hi = torch.zeros_like(rd), torch.full_like(rd, pmax)
        inv = rd <= _kb(k, pmax)
        for _ in range(60):
            mid = 0.5 * (lo + hi)
            up = _kb(k, mid) < rd
            lo, hi = torch.where(up, mid, lo), torch.where(up, hi, mid)
        p = 0.5 * (lo + hi)
        q = torch.where(rd > 0, p.sin() / rd.clamp(min=1e-300), torch.zeros_like(rd))
        dx, dy, dz = q * uu, q * vv, p.cos()
    th, ph = torch.atan2(dx, dz), torch.atan(dy / dz)
    ub, vb = th / fx * w + 0.5 * w - 0.5, ph / fy * h + 0.5 * h - 0.5
    inside = inv & (ub >= -0.5) & (ub <= w - 0.5) & (vb >= -0.5) & (vb <= h - 0.5)
    native = torch.where(inside[..., None], _bilinear(beap, torch.where(inside, ub, z), torch.where(inside, vb, z)), z)
    cen = (th.abs() <= 0.5 * w / f) & (ph.abs() <= 0.5 * h / f)
    # SSIM with an 11 x 11 Gaussian window, and squared errors, per region
    g1 = torch.exp(-torch.arange(-5, 6, device="cuda", dtype=F64) ** 2 / (2 * 1.5 ** 2))
    g1 = (g1 / g1.sum()).view(1, 1, 1, 11)

    def blur(a):
        a = torch.nn.functional.conv2d(a[:, None], g1, padding=(0, 5))
        return torch.nn.functional.conv2d(a, g1.transpose(2, 3), padding=(5, 0))[:, 0]

    a, b = native.permute(2, 0, 1).contiguous(), gt.permute(2, 0, 1).contiguous()
    ma, mb = blur(a), blur(b)
    va, vb2, cab = blur(a * a) - ma * ma, blur(b * b) - mb * mb, blur(a * b) - ma * mb
    c1, c2 = 0.01 ** 2, 0.03 ** 2
    ssim = ((2 * ma * mb + c1) * (2 * cab + c2) / ((ma * ma + mb * mb + c1) * (va + vb2 + c2))).mean(0)
    se = ((a - b) ** 2).sum(0)
    met = [[float(se[m].sum()), float(ssim[m].sum()), None] for m in (inside & cen, inside & ~cen)]
    return {"supervision": sup, "valid": None, "native": native, "regions": None, "metrics": met}


def exact(case, seed):
    kind = case["kind"]
    if kind == "evaluate":
        return _evaluate64(prepare(case, seed))
    if kind == "optimise":
        s = prepare(case, seed)
        a, n = s["adam"], case["n"]
        K3 = 3 * (case["deg"] + 1) ** 2
        f32 = lambda v: float(np.float32(v))  # noqa: E731
        b1, b2, eps = f32(a.hp["beta1"]), f32(a.hp["beta2"]), f32(a.hp["eps"])
        t = a.t + 1
        out, ms, vs, off = {}, [], [], 0
        for r, k, lr in (("mean", "mean", "lr_mean"), ("log_scale", "scale", "lr_scale"), ("quat", "quat", "lr_quat"),
                         ("logit_opacity", "opacity", "lr_opacity"), ("sh", "sh", None)):
            x, gr = a.raw[r].to(F64), s["grads"][k].to(F64)
            if r == "log_scale":
                gr = gr * x.exp()
            elif r == "logit_opacity":
                gr = gr * torch.sigmoid(x) * (1 - torch.sigmoid(x))
            m, v = (q[off:off + x.numel()].to(F64).view_as(x) for q in (a.m, a.v))
            off += x.numel()
            m, v = b1 * m + (1 - b1) * gr, b2 * v + (1 - b2) * gr * gr
            rate = f32(a.hp[lr]) if lr else torch.tensor([f32(a.hp["lr_sh_dc"])] * 3 + [f32(a.hp["lr_sh_rest"])] * (K3 - 3),
                                                         dtype=F64, device="cuda").view(1, K3 // 3, 3)
            out[r] = x - rate * (m / (1 - b1 ** t)) / ((v / (1 - b2 ** t)).sqrt() + eps)
            ms.append(m.reshape(-1))
            vs.append(v.reshape(-1))
        assert off == n * (11 + K3)
        return {**out, "m": torch.cat(ms), "v": torch.cat(vs), "scale": out["log_scale"].exp(),
                "opacity": torch.sigmoid(out["logit_opacity"])}
    if kind in ("view", "stream", "noalloc", "autograd", "train"):
        pairs = case["n"] * case["w"] * case["h"]
        if case.get("splat") or case.get("cams", 1) > 1 or pairs > (2 << 30) or (kind in ("train", "autograd") and pairs > (1 << 24)):
            return None  # every ray against every Gaussian takes too long there, or too much memory to differentiate
        s = prepare(case, seed)
        cam = _camera(case)
        if _geometry(cam)[1] is None:
            return None
        p = [getattr(s["g"], k).to(F64) for k in NAMES]
        if kind in ("view", "stream", "noalloc"):
            rgb, T = _render64(cam, *p, case["deg"])
            return [rgb, T] if kind == "noalloc" else rgb
        p = [t.requires_grad_(True) for t in p]
        rgb, _ = _render64(cam, *p, case["deg"])
        loss = (rgb - s["target"].to(F64)).abs().mean()
        loss.backward()
        return {"rgb": rgb.detach(), "loss": loss.detach() if kind == "autograd" else loss.detach().view(1),
                **{k: t.grad for k, t in zip(NAMES, p)}}
    return None
