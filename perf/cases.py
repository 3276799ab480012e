"""What is measured of this renderer: one dict per case, through the package's public entry points.

Kinds of case, and what each stands for:

* frame        one relit frame (Renderer.render): a viewer or an offline renderer moving camera and light;
* fixed_light  a new view under the light of the frame before (Renderer.render_stages without the light splat);
* environment  one frame under several directional lights (Renderer.render_environment);
* train        one training view: render, L1 + D-SSIM loss with its image gradient, backward to every parameter (the
               loss sees a stored image in place of this pass's own render: its |x - y| has a kink, and a last-bit
               difference of the render would turn single pixels' gradients round);
* adam         the optimiser's step over every parameter group of a scene;
* serve        a burst of requests of two scenes and several resolutions through the server;
* order        the depth sort alone, for callers that may not allocate device memory.

Scenes follow the distributions of paper_2410_11419_gb300.synth (noisy sphere shell plus 10 % fluff, or a ball;
log-uniform scales; K lobes per Gaussian or one shared basis; Xavier MLPs), drawn on the GPU so that inputs are quick
to make.  `exact` restates the frame, the loss and their gradients in float64 with plain torch operations.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch
import torch.nn.functional as F
from torch.utils.checkpoint import checkpoint

from paper_2410_11419_gb300 import _native as N
from paper_2410_11419_gb300 import render as R
from paper_2410_11419_gb300 import synth
from paper_2410_11419_gb300.train import LOWER_BOUND, Schedule

DTYPES = {"fp32": N.GS3_MLP_FP32, "bf16": N.GS3_MLP_BF16, "fp8": N.GS3_MLP_FP8_E4M3}
CAMERA_SIDE = N.GS3_STAGE_PREP | N.GS3_STAGE_CAMERA_BIN | N.GS3_STAGE_MLP | N.GS3_STAGE_CAMERA
LAMBDA = 0.2  # weight of the D-SSIM term
BETAS, EPS, STEP = (0.9, 0.999), 1e-15, 1000  # the trainer's Adam, some way into a run

# (phi width, phi layers, psi width, psi layers, activation) of the networks in use
NETS = {
    "tiny": (64, 2, 64, 2, synth.RELU),       # the 1,000-Gaussian scene
    "object": (128, 3, 128, 3, synth.RELU),   # the object scenes and the serving mix
    "paper": (32, 3, 128, 3, synth.LEAKY_RELU),
    "narrow": (16, 2, 32, 2, synth.RELU),     # FP32 only
}


def _case(kind, n, width, height, k=8, shape="shell", net="object", mlp="bf16", light="point", shared=False,
          lights=1, requests=1, ablate=0):
    return dict(kind=kind, n=n, width=width, height=height, k=k, shape=shape, net=net, mlp=mlp, light=light,
                shared=shared, lights=lights, requests=requests, ablate=ablate)


def listed():
    cases = {
        # the smallest frame a user renders (previews, unit scenes): launches and latency
        "tiny_frame_fp32": _case("frame", 1000, 128, 128, k=4, shape="ball", net="tiny", mlp="fp32"),
        # a captured object at the paper's smallest size, with the paper's networks in full precision
        "paper_frame_fp32": _case("frame", 120_000, 512, 512, net="paper", mlp="fp32"),
        # the benchmark workload: one relit frame of the 300k object at 800x800
        "object_frame_bf16": _case("frame", 300_000, 800, 800),
        # the largest scene of the serving mix at its largest resolution
        "large_frame_bf16": _case("frame", 1_000_000, 1024, 1024),
        # sunlight on a mid-sized scene: ragged image, FP8 networks, one shared lobe basis
        "sun_frame_fp8": _case("frame", 250_000, 747, 501, mlp="fp8", light="directional", shared=True),
        # turning the camera around an object under a fixed light
        "moving_camera_bf16": _case("fixed_light", 300_000, 800, 800),
        # image-based lighting with eight directions
        "environment_bf16": _case("environment", 100_000, 512, 512, light="directional", lights=8),
        # one training view of the benchmark workload
        "train_object_fp32": _case("train", 300_000, 800, 800, mlp="fp32"),
        # one training view of a small scene with the paper's networks, early in the schedule (no lobes yet)
        "train_small_fp32": _case("train", 20_000, 256, 256, net="paper", mlp="fp32",
                                  ablate=N.GS3_ABLATE_SPECULAR),
        # the optimiser's step that follows each training view
        "adam_object": _case("adam", 300_000, 16, 16, mlp="fp32"),
        # a burst of eight requests: 100k and 250k scenes, three resolutions, four in flight
        "serve_mix_bf16": _case("serve", 100_000, 800, 800, requests=8),
        # the depth order of the benchmark scene for an embedding renderer
        "order_300k": _case("order", 300_000, 16, 16),
    }
    return [dict(c, name=name) for name, c in cases.items()]


def draw(rng):
    def spread(lo, hi):
        return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    def size(hi):
        h = spread(96, hi)
        return min(hi, max(64, int(h * rng.uniform(0.6, 1.7)))), h

    kind = rng.choice(["frame"] * 5 + ["fixed_light", "environment", "train", "train", "adam", "serve", "order"])
    k = rng.choice([1, 4, 8, 8, 8, 16])
    shape = rng.choice(["ball", "shell", "shell", "shell"])
    shared = rng.random() < 0.25
    light = "directional" if rng.random() < 0.25 else "point"
    mlp = rng.choice(["fp32", "bf16", "bf16", "fp8"])
    net = rng.choice(["tiny", "object", "object", "paper"] + (["narrow"] if mlp == "fp32" else []))
    shell = shape == "shell"  # few rays end early in a full ball: the same cost at fewer Gaussians
    more = dict(k=k, shape=shape, shared=shared, net=net, mlp=mlp, light=light)
    if kind in ("frame", "fixed_light"):
        w, h = size(1024)
        return _case(kind, spread(500, 1_000_000 if shell else 250_000), w, h, **more)
    if kind == "environment":
        w, h = size(512)
        return _case(kind, spread(500, 100_000 if shell else 40_000), w, h, lights=rng.randint(2, 8),
                     **dict(more, light="directional"))
    if kind == "train":
        w, h = size(800)
        return _case(kind, spread(500, 300_000 if shell else 20_000), w, h,
                     ablate=rng.choice([0, 0, N.GS3_ABLATE_SPECULAR]), **more)
    if kind == "adam":
        return _case(kind, spread(500, 300_000), 16, 16, k=k, shape=shape, shared=shared, net=net, mlp="fp32")
    if kind == "serve":
        w, h = size(800)
        return _case(kind, spread(1000, 100_000 if shell else 40_000), w, h, requests=rng.randint(3, 8), **more)
    return _case(kind, spread(500, 1_000_000), 16, 16)


# -- inputs -------------------------------------------------------------------

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(1_000_003 * seed + 17)


def _scene(case, n, seed):
    """A host scene (synth.Scene) with synth's distributions, drawn on the GPU."""
    g, k = _generator(seed), case["k"]

    def normal(*shape):
        return torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)

    def uniform(*shape):
        return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)

    def unit(x):
        return x / x.norm(dim=-1, keepdim=True)

    def host(x, pad=0):
        return F.pad(x, (0, pad)).float().cpu().numpy()

    if case["shape"] == "ball":
        pos = unit(normal(n, 3)) * uniform(n, 1) ** (1 / 3)
    else:
        fluff = n // 10
        shell = unit(normal(n - fluff, 3)) * (1 + 0.02 * normal(n - fluff, 1))
        pos = torch.cat([shell, unit(normal(fluff, 3)) * uniform(fluff, 1) ** (1 / 3)])
    scale = torch.exp(math.log(0.01) + math.log(8.0) * uniform(n, 3))
    rot, logit, albedo, shade = unit(normal(n, 4)), normal(n, 1), uniform(n, 3), unit(normal(n, 4))
    latent = 0.1 * normal(n, 6)
    m = 1 if case["shared"] else n
    if case["shared"]:
        lobe_rot = unit(normal(k, m, 4))
        sxy = 0.3 + 0.7 * uniform(k, m, 2)
    else:  # the minimal rotation from e_z to a uniform axis; isotropic lobes
        a = unit(normal(k, m, 3))
        lobe_rot = unit(torch.stack([1 + a[..., 2], -a[..., 1], a[..., 0], torch.zeros_like(a[..., 0])], -1))
        sxy = torch.ones(k, m, 2, device="cuda", dtype=torch.float64)
    sz = torch.exp(math.log(100.0) * uniform(k, m, 1)) ** -0.5
    pw, ph, sw, sh, act = NETS[case["net"]]
    return synth.Scene(
        n=n, k=k, mean_op=host(torch.cat([pos, logit], 1)), scale=host(scale, 1), rot=host(rot),
        shade_rot=host(shade), albedo_d=host(albedo, 1), albedo_s=host(torch.ones_like(albedo), 1),
        latent=host(torch.stack([latent[:, :4], F.pad(latent[:, 4:], (0, 2))])),
        lobe_rot=host(lobe_rot), lobe_sigma=host(torch.cat([sxy, sz], -1), 1),
        lobe_amp=host(0.5 * uniform(k, n, 3), 1),
        phi=synth.make_mlp(seed, "phi", 61, pw, ph, 1, act), psi=synth.make_mlp(seed, "psi", 60, sw, sh, 3, act),
        lobe_shared=case["shared"])


def _view(case, seed, width=None, height=None):
    width, height = width or case["width"], height or case["height"]
    cam, light = synth.camera_light_pair(seed, width, height)
    return cam, synth.directional_light(seed) if case["light"] == "directional" else light


def _images(case, seed):
    """A smooth photograph in [0, 1] and a darker, noisy render of it."""
    g, w, h = _generator(seed + 5), case["width"], case["height"]
    y, x = (torch.arange(h, device="cuda") / h)[:, None, None], (torch.arange(w, device="cuda") / w)[None, :, None]
    f, ph = 2 + 10 * torch.rand(2, 3, generator=g, device="cuda"), 6.28 * torch.rand(3, generator=g, device="cuda")
    photo = (0.5 + 0.4 * torch.sin(f[0] * x + ph) * torch.cos(f[1] * y)).contiguous()
    noise = torch.randn(photo.shape, generator=g, device="cuda")
    return photo, (0.9 * photo + 0.1 * noise).clamp(min=0)


def _renderer(ds, cam, lights, width, height):
    """A renderer whose pair capacity holds this view (every splat binned once, 5 % head room)."""
    probe, need = R.Renderer(ds, width, height, 1), 1
    for light in lights:
        probe.render_stages(cam, light, N.GS3_STAGE_PREP | N.GS3_STAGE_CAMERA_BIN | N.GS3_STAGE_LIGHT_BIN)
        head = probe.header()
        need = max(need, head.pairs_cam_needed, head.pairs_light_needed)
    return R.Renderer(ds, width, height, need + need // 20 + 1024)


def _requests(case, seed):
    """(scene index, width, height, view seed) of a burst: the case's size, 5/8 and 8/25 of it, two scenes in turn."""
    w, h = case["width"], case["height"]
    sizes = [(w, h), (max(16, w * 16 // 25), max(16, h * 16 // 25)), (max(16, w * 8 // 25), max(16, h * 8 // 25))]
    return [(i % 2, *sizes[i % 3], seed + 31 * i) for i in range(case["requests"])]


def _scenes(case, seed):
    if case["kind"] == "serve":
        return [_scene(case, case["n"], seed), _scene(case, case["n"] * 5 // 2, seed + 1)]
    return [_scene(case, case["n"], seed)]


def _adam_state(case, seed):
    scene = _scene(case, case["n"], seed)
    p = {f: torch.from_numpy(np.ascontiguousarray(getattr(scene, f))).cuda() for f in scene.ARRAYS}
    for name in ("phi", "psi"):
        w, b = getattr(scene, name).packed()
        p[name + "_w"], p[name + "_b"] = torch.from_numpy(w).cuda(), torch.from_numpy(b).cuda()
    g = _generator(seed + 7)
    grad = {f: 1e-4 * torch.randn(x.shape, generator=g, device="cuda") for f, x in p.items()}
    m = {f: 1e-4 * torch.randn(x.shape, generator=g, device="cuda") for f, x in p.items()}
    v = {f: 1e-8 * torch.rand(x.shape, generator=g, device="cuda") for f, x in p.items()}
    return p, grad, m, v


def _keys(case, seed):
    """FP32 depths of Gaussians seen from radius 3, as their bit patterns."""
    d = 2 + 2 * torch.rand(case["n"], generator=_generator(seed), device="cuda")
    return d.view(torch.int32)


def prepare(case, seed):
    kind = case["kind"]
    s = SimpleNamespace(kind=kind)
    if kind == "adam":
        s.p, s.grad, s.m, s.v = _adam_state(case, seed)
        s.schedule = Schedule()
        return s
    if kind == "order":
        s.keys = _keys(case, seed)
        s.out = torch.empty_like(s.keys)
        return s
    dev = [R.DeviceScene(x, mlp_dtype=DTYPES[case["mlp"]]) for x in _scenes(case, seed)]
    if kind == "serve":
        s.server = R.Server(hbm_budget=16 << 30, max_inflight=4)
        ids = [s.server.add_scene(x) for x in dev]
        s.requests = [(ids[i], *_view(case, vs, w, h), torch.empty((h, w, 3), device="cuda"))
                      for i, w, h, vs in _requests(case, seed)]
        torch.cuda.synchronize()
        return s
    s.cam, s.light = _view(case, seed)
    lights = [s.light]
    if kind == "environment":
        s.lights, s.weights = synth.environment_lights(seed, case["lights"])
        lights = s.lights
    s.rd = _renderer(dev[0], s.cam, lights, case["width"], case["height"])
    if kind == "fixed_light":  # the frame whose light stays
        s.rd.render(_view(case, seed + 1)[0], s.light)
    if kind == "train":
        s.photo, s.seen = _images(case, seed)
        s.opts = R.opts_struct(ablate=case["ablate"])
    return s


def run(s):
    if s.kind == "frame":
        return s.rd.render(s.cam, s.light)
    if s.kind == "fixed_light":
        return s.rd.render_stages(s.cam, s.light, CAMERA_SIDE)
    if s.kind == "environment":
        return s.rd.render_environment(s.cam, s.lights, s.weights)
    if s.kind == "train":
        img = s.rd.render(s.cam, s.light, s.opts)
        loss, dimg = R.loss_l1_dssim(s.seen, s.photo, LAMBDA)
        return {"image": img, "loss": loss, "dimg": dimg, "grads": s.rd.backward(s.cam, s.light, dimg, s.opts)}
    if s.kind == "adam":
        stream = torch.cuda.current_stream().cuda_stream
        for f in N.GRAD_FIELDS:
            N.gs3_adam_step(s.p[f], s.grad[f], s.m[f], s.v[f], s.schedule.lr(f, STEP), BETAS[0], BETAS[1], EPS, STEP,
                            LOWER_BOUND.get(f, -math.inf), stream)
        return {"p": s.p, "m": s.m, "v": s.v}
    if s.kind == "serve":
        tickets = [s.server.submit(*r) for r in s.requests]
        for t in tickets:
            status, _ = s.server.wait(t)
            if status != N.GS3_OK:
                raise RuntimeError(f"request failed: {N.STATUS_NAMES.get(status, status)}")
        return [r[3] for r in s.requests]
    N.gs3_depth_order_static(s.keys, s.keys.numel(), s.out, torch.cuda.current_stream().cuda_stream)
    return s.out


# -- what a pass cannot do without -------------------------------------------

def _params(case, n):
    """Floats of the per-Gaussian arrays and of the networks' weights."""
    per = 4 * (8 + case["k"] * (1 if case["shared"] else 3))
    pw, ph, sw, sh, _ = NETS[case["net"]]
    net = sum(a * b + b for w, l, i, o in ((pw, ph, 61, 1), (sw, sh, 60, 3))
              for a, b in zip([i] + [w] * l, [w] * l + [o]))
    return n * per, net


def _frame_work(case, n, width, height, lights=1, shadow=True):
    pw, ph, sw, sh, _ = NETS[case["net"]]
    phi = 2 * (61 * pw + (ph - 1) * pw * pw + pw)
    psi = 2 * (60 * sw + (sh - 1) * sw * sw + 3 * sw)
    # a Gaussian's alpha >= 1/255 ellipse covers 0.0358 (f / 3)^2 pixels in the mean over the scenes' scales and
    # rotations (f the focal length in pixels, 1.374 height); 12 operations per covered light pixel
    cover = 12.0 * n * 0.0358 * (1.374 * height / 3) ** 2 if shadow else 0.0
    per, net = _params(case, n)
    return {"bytes": 4.0 * (per + net) + 12.0 * width * height, "flops": n * (phi * lights + psi) + lights * cover}


def work(case):
    kind, n, w, h = case["kind"], case["n"], case["width"], case["height"]
    if kind == "adam":
        per, net = _params(case, n)
        return {"bytes": 28.0 * (per + net), "flops": 12.0 * (per + net)}
    if kind == "order":
        return {"bytes": 8.0 * n, "flops": 0.0}
    if kind == "serve":
        each = [_frame_work(case, (n, n * 5 // 2)[i], rw, rh) for i, rw, rh, _ in _requests(case, 0)]
        return {f: sum(x[f] for x in each) for f in ("bytes", "flops")}
    one = _frame_work(case, n, w, h, case["lights"], kind != "fixed_light")
    if kind == "train":  # parameters in and gradients out, image, target and image gradient; backward twice the forward
        return {"bytes": 2 * one["bytes"] + 12.0 * w * h, "flops": 3 * one["flops"]}
    return one


# -- the same results in float64, by plain torch -------------------------------

D = torch.float64
AMIN, AMAX, TSTOP = (float(np.float32(x)) for x in (1 / 255, 0.99, 1e-4))
LOWPASS, BIAS, NEAR, FRUSTUM = float(np.float32(0.3)), np.float32(0.015), float(np.float32(0.2)), 1.3


def _dev(x, dtype=D):
    return torch.as_tensor(np.asarray(x), device="cuda").to(dtype)


def _rot(q):
    w, x, y, z = (q / q.norm(dim=-1, keepdim=True)).unbind(-1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], -1).unflatten(-1, (3, 3))


def _light_view(light, width, height):
    """FP32 rotation and translation of the light's view (it looks at the origin, +z up), and its pixels per unit if
    orthographic, else 0."""
    f32, ortho = np.float32, 0.0
    eye = np.asarray(light.pos, f32)
    if light.type == 1:
        eye = np.asarray(light.dir, f32) * (f32(4) * f32(light.extent))
        ortho = float(f32(0.5) * f32(min(width, height)) / f32(light.extent))

    def dot(a, b):
        return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]

    def cross(a, b):
        return np.array([a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]], f32)

    fwd = -eye / np.sqrt(dot(eye, eye))
    up = np.array([0, 0, 1] if abs(fwd[2]) <= f32(0.999) else [0, 1, 0], f32)
    right = cross(fwd, up)
    right = right / np.sqrt(dot(right, right))
    rot = np.stack([right, cross(fwd, right), fwd])
    return rot, np.array([-dot(r, eye) for r in rot], f32), ortho


def _project(P, rot, t, cam, ortho):
    """Screen positions, conics, and the tiles of every Gaussian in one view, in lists ordered by FP32 depth."""
    mu, logit = P["mean_op"][:, :3], P["mean_op"][:, 3]
    Rv, tv = _dev(rot), _dev(t)
    p = mu @ Rv.T + tv
    x, y, z = p.unbind(1)
    zero = torch.zeros_like(z)
    if ortho:
        u, v = ortho * x + cam.cx, ortho * y + cam.cy
        s = torch.full_like(z, ortho)
        J = torch.stack([s, zero, zero, zero, s, zero], 1).unflatten(1, (2, 3))
        limx, limy, sx, sy = FRUSTUM * 0.5 * cam.width / ortho, FRUSTUM * 0.5 * cam.height / ortho, x, y
    else:
        u, v = cam.fx * x / z + cam.cx, cam.fy * y / z + cam.cy
        J = torch.stack([cam.fx / z, zero, -cam.fx * x / (z * z), zero, cam.fy / z, -cam.fy * y / (z * z)],
                        1).unflatten(1, (2, 3))
        limx, limy, sx, sy = FRUSTUM * 0.5 * cam.width / cam.fx, FRUSTUM * 0.5 * cam.height / cam.fy, x / z, y / z
    M = J @ Rv @ (_rot(P["rot"]) * P["scale"][:, None, :3])
    C = M @ M.transpose(1, 2)
    a, b, c = C[:, 0, 0] + LOWPASS, C[:, 0, 1], C[:, 1, 1] + LOWPASS
    det = a * c - b * b
    with torch.no_grad():
        r = torch.ceil(3 * torch.sqrt((a + c) / 2 + torch.sqrt(((a + c) ** 2 / 4 - det).clamp(min=0.1))))
        r2 = 2 * (logit.clamp(max=0) - math.log(AMIN))
        hx, hy = torch.sqrt(r2.clamp(min=0) * a), torch.sqrt(r2.clamp(min=0) * c)
        gx, gy = -(-cam.width // 16), -(-cam.height // 16)
        x0, x1 = torch.floor((u - torch.minimum(r, hx)) / 16), torch.floor((u + torch.minimum(r, hx)) / 16)
        y0, y1 = torch.floor((v - torch.minimum(r, hy)) / 16), torch.floor((v + torch.minimum(r, hy)) / 16)
        keep = (z > NEAR) & (sx.abs() <= limx) & (sy.abs() <= limy) & (r2 > 0)
        keep &= (x1 >= 0) & (x0 < gx) & (y1 >= 0) & (y0 < gy)
        x0, x1, y0, y1 = x0.clamp(min=0), x1.clamp(max=gx - 1), y0.clamp(min=0), y1.clamp(max=gy - 1)
    return SimpleNamespace(uv=torch.stack([u, v], 1), conic=torch.stack([c / det, -b / det, a / det], 1), gx=gx, gy=gy,
                           rect=[q.long() for q in (x0, x1, y0, y1)], keep=keep)


def _lists(view, key):
    """Gaussians of each tile in the order of their FP32 keys (ties by index): one long list and the tiles' starts."""
    order = torch.argsort(key, stable=True)
    order = order[view.keep[order]]
    x0, x1, y0, y1 = (q[order] for q in view.rect)
    count = (x1 - x0 + 1) * (y1 - y0 + 1)
    which = torch.repeat_interleave(torch.arange(len(order), device="cuda"), count)
    i = torch.arange(len(which), device="cuda") - (torch.cumsum(count, 0) - count)[which]
    w = (x1 - x0 + 1)[which]
    tile = (y0[which] + i // w) * view.gx + x0[which] + i % w
    tile, at = torch.sort(tile, stable=True)
    starts = torch.searchsorted(tile, torch.arange(view.gx * view.gy + 1, device="cuda"))
    return order[which[at]], starts.tolist()


def _pixels(t, gx, cam):
    xs = torch.arange(t % gx * 16, min(cam.width, t % gx * 16 + 16), device="cuda")
    ys = torch.arange(t // gx * 16, min(cam.height, t // gx * 16 + 16), device="cuda")
    return (ys[:, None] * cam.width + xs[None]).reshape(-1)


def _alpha(uv, conic, gamma, lst, pix, cam):
    dx = (pix % cam.width + 0.5)[:, None] - uv[lst, 0]
    dy = (pix // cam.width + 0.5)[:, None] - uv[lst, 1]
    A, B, C = conic[lst].unbind(1)
    beta = torch.exp(-0.5 * (A * dx * dx + C * dy * dy) - B * dx * dy)
    alpha = (gamma[lst] * beta).clamp(max=AMAX)
    return beta, torch.where(alpha.detach() >= AMIN, alpha, 0.0)


def _tilewise(fn, grad, *args):
    return checkpoint(fn, *args, use_reentrant=False) if grad else fn(*args)


def _shadow(P, cam, light, grad):
    """T of every Gaussian: its beta-weighted mean transmittance over the light's pixels (bias 0.015)."""
    rot, t, ortho = _light_view(light, cam.width, cam.height)
    view = _project(P, rot, t, cam, ortho)
    m32 = P["mean_op"].detach().float()
    if light.type == 1:
        r, tt = _dev(rot, torch.float32), _dev(t, torch.float32)
        key = r[2, 0] * m32[:, 0] + r[2, 1] * m32[:, 1] + r[2, 2] * m32[:, 2] + tt[2]
    else:
        d = m32[:, :3] - _dev(light.pos, torch.float32)
        key = torch.sqrt(d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1] + d[:, 2] * d[:, 2])
    lists, starts = _lists(view, key)
    gamma = torch.sigmoid(P["mean_op"][:, 3])

    def tile(uv, conic, gamma, lst, pix):
        beta, alpha = _alpha(uv, conic, gamma, lst, pix, cam)
        log = F.pad(torch.cumsum(torch.log1p(-alpha), 1), (1, 0))
        dist = key[lst]
        occluders = torch.searchsorted(dist, dist - float(BIAS))
        beta = torch.where(alpha.detach() > 0, beta, 0.0)
        return (beta * torch.exp(log[:, occluders])).sum(0), beta.sum(0)

    parts = [(lists[b:e], *_tilewise(tile, grad, view.uv, view.conic, gamma, lists[b:e], _pixels(k, view.gx, cam)))
             for k, (b, e) in enumerate(zip(starts, starts[1:])) if e > b]
    num = den = torch.zeros_like(gamma)
    if parts:
        ids = torch.cat([q[0] for q in parts])
        num, den = (torch.zeros_like(gamma).index_add(0, ids, torch.cat([q[i] for q in parts])) for i in (1, 2))
    return torch.where(den > 0, num / torch.where(den > 0, den, 1.0), 1.0)


def _directions(P, cam, light):
    mu = P["mean_op"][:, :3]
    to = _dev(light.pos) - mu if light.type == 0 else _dev(light.dir).expand_as(mu)
    out = _dev(cam.pos) - mu
    return to, to / to.norm(dim=1, keepdim=True), out / out.norm(dim=1, keepdim=True)


def _shade(P, cam, light, ablate):
    """Modified Lambertian term plus angular-Gaussian lobes, times the light's irradiance."""
    to, wi, wo = _directions(P, cam, light)
    Rs = _rot(P["shade_rot"])
    wi, wo = (Rs @ wi[:, :, None])[..., 0], (Rs @ wo[:, :, None])[..., 0]
    off, x = 0.01 * (1 - math.exp(-1)), wi[:, 2]
    fd = (torch.where(x > 0, x, 0.01 * torch.expm1(x.clamp(max=0))) + off) / ((1 + off) * math.pi)
    h = wi + wo
    h = h / h.norm(dim=1, keepdim=True)
    fs = torch.zeros_like(h)
    for j in range(0 if ablate & N.GS3_ABLATE_SPECULAR else P["lobe_amp"].shape[0]):
        l = (_rot(P["lobe_rot"][j]).transpose(1, 2) @ h[:, :, None])[..., 0]
        sig, sxy = P["lobe_sigma"][j], torch.sqrt(l[:, 0] ** 2 + l[:, 1] ** 2)
        q = (l[:, 0] / sxy / sig[:, 0]) ** 2 + (l[:, 1] / sxy / sig[:, 1]) ** 2
        G = torch.exp(-0.5 * torch.atan2(sxy, l[:, 2]) ** 2 * q / sig[:, 2] ** 2) / sig[:, 2]
        fs = fs + P["lobe_amp"][j][:, :3] * G[:, None]
    E = light.intensity / (to * to).sum(1, keepdim=True) if light.type == 0 else light.intensity
    return E * (P["albedo_d"][:, :3] * fd[:, None] + P["albedo_s"][:, :3] * fs)


def _encode(v):
    return torch.cat([v] + [f(2.0 ** q * math.pi * v) for q in range(4) for f in (torch.sin, torch.cos)], 1)


def _network(w, b, net, x):
    wo = bo = 0
    dims = net.dims()
    for i, (fi, fo) in enumerate(dims):
        x = x @ w[wo:wo + fi * fo].view(fo, fi).T + b[bo:bo + fo]
        wo, bo = wo + fi * fo, bo + fo
        if i + 1 < len(dims):
            x = F.relu(x) if net.act == synth.RELU else F.leaky_relu(x, 0.01)
    return torch.sigmoid(x)


def _composite(P, cam, cols, grad):
    """Channels `cols` [N, c] composited toward the camera; a ray stops before T falls below 1e-4."""
    view = _project(P, cam.R, cam.t, cam, 0.0)
    m32, r, t = P["mean_op"].detach().float(), _dev(cam.R, torch.float32), _dev(cam.t, torch.float32)
    lists, starts = _lists(view, r[2, 0] * m32[:, 0] + r[2, 1] * m32[:, 1] + r[2, 2] * m32[:, 2] + t[2])
    gamma = torch.sigmoid(P["mean_op"][:, 3])

    def tile(uv, conic, gamma, cols, lst, pix):
        _, alpha = _alpha(uv, conic, gamma, lst, pix, cam)
        log = torch.log1p(-alpha)
        through = torch.cumsum(log, 1)
        stop = (alpha.detach() > 0) & (torch.exp(through.detach()) < TSTOP)
        on = torch.cumsum(stop, 1) == 0
        return torch.where(on, alpha * torch.exp(through - log), 0.0) @ cols[lst]

    ids, vals = [], []
    for k, (b, e) in enumerate(zip(starts, starts[1:])):
        if e > b:
            ids.append(_pixels(k, view.gx, cam))
            vals.append(_tilewise(tile, grad, view.uv, view.conic, gamma, cols, lists[b:e], ids[-1]))
    img = torch.zeros(cam.width * cam.height, cols.shape[1], device="cuda", dtype=D)
    img = img.index_copy(0, torch.cat(ids), torch.cat(vals)) if ids else img
    return img.unflatten(0, (cam.height, cam.width))


def _parameters(scene, grad):
    P = {f: _dev(getattr(scene, f)) for f in scene.ARRAYS}
    for name in ("phi", "psi"):
        w, b = getattr(scene, name).packed()
        P[name + "_w"], P[name + "_b"] = _dev(w), _dev(b)
    return {f: x.requires_grad_(grad) for f, x in P.items()}


def _image(P, scene, cam, lights, weights, ablate=0, grad=False):
    mu = P["mean_op"][:, :3]
    rest = torch.cat([_encode(mu), P["latent"][0], P["latent"][1][:, :2]], 1)
    cols, wo = [], _directions(P, cam, lights[0])[2]
    cols.append(_network(P["psi_w"], P["psi_b"], scene.psi, torch.cat([_encode(wo), rest], 1)))
    for light in lights:
        T, wi = _shadow(P, cam, light, grad), _directions(P, cam, light)[1]
        phi = _network(P["phi_w"], P["phi_b"], scene.phi, torch.cat([T[:, None], _encode(wi), rest], 1))
        cols += [_shade(P, cam, light, ablate), phi]
    out = _composite(P, cam, torch.cat(cols, 1), grad)
    return sum(w * (out[..., 3 + 4 * i:6 + 4 * i] * out[..., 6 + 4 * i:7 + 4 * i] + out[..., :3])
               for i, w in enumerate(weights))


def _loss(img, target):
    g = torch.exp(-(torch.arange(11, device="cuda", dtype=D) - 5) ** 2 / (2 * 1.5 ** 2))
    g = g / g.sum()

    def blur(x):
        x = F.conv2d(x[:, None], g.view(1, 1, 1, 11), padding=(0, 5))
        return F.conv2d(x, g.view(1, 1, 11, 1), padding=(5, 0))[:, 0]

    x, y = img.permute(2, 0, 1), target.permute(2, 0, 1)
    mx, my = blur(x), blur(y)
    sxx, syy, sxy = blur(x * x) - mx * mx, blur(y * y) - my * my, blur(x * y) - mx * my
    c1, c2 = 0.01 ** 2, 0.03 ** 2
    ssim = (2 * mx * my + c1) * (2 * sxy + c2) / ((mx * mx + my * my + c1) * (sxx + syy + c2))
    return (1 - LAMBDA) * (x - y).abs().mean() + LAMBDA * (1 - ssim.mean())


def exact(case, seed):
    kind = case["kind"]
    if kind == "order":
        return None  # whole numbers
    if kind == "adam":
        p, grad, m, v = ({f: x.to(D) for f, x in d.items()} for d in _adam_state(case, seed))
        b1, b2 = (float(np.float32(b)) for b in BETAS)
        for f in p:
            m[f] = b1 * m[f] + (1 - b1) * grad[f]
            v[f] = b2 * v[f] + (1 - b2) * grad[f] ** 2
            step = Schedule().lr(f, STEP) * (m[f] / (1 - b1 ** STEP)) / (torch.sqrt(v[f] / (1 - b2 ** STEP)) + EPS)
            p[f] = (p[f] - step).clamp(min=LOWER_BOUND.get(f, -math.inf))
        return {"p": p, "m": m, "v": v}
    scenes = _scenes(case, seed)
    if kind == "train":
        cam, light = _view(case, seed)
        P = _parameters(scenes[0], True)
        img = _image(P, scenes[0], cam, [light], [1.0], case["ablate"], True)
        photo, seen = (x.to(D) for x in _images(case, seed))
        loss = _loss(seen.requires_grad_(True), photo)
        dimg, = torch.autograd.grad(loss, seen)
        img.backward(dimg)
        grads = {f: P[f].grad if P[f].grad is not None else torch.zeros_like(P[f]) for f in N.GRAD_FIELDS}
        return {"image": img.detach(), "loss": loss.detach()[None], "dimg": dimg, "grads": grads}
    with torch.no_grad():
        params = [_parameters(x, False) for x in scenes]
        if kind == "serve":
            return [_image(params[i], scenes[i], cam, [light], [1.0])
                    for i, w, h, vs in _requests(case, seed) for cam, light in [_view(case, vs, w, h)]]
        cam, light = _view(case, seed)
        if kind == "environment":
            lights, weights = synth.environment_lights(seed, case["lights"])
            return _image(params[0], scenes[0], cam, lights, [float(w) for w in weights])
        return _image(params[0], scenes[0], cam, [light], [1.0])
