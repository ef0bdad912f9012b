"""The rasterizer's work as its users call it, for timing and for comparing two
versions of the library: listed cases, random cases of the same ranges, their
inputs (made on the GPU from a seed), one pass through the public entry points,
the bytes a pass cannot do without, and its outputs in 64-bit arithmetic.

Kinds of case
  step    adop_render_forward + adop_render_backward of one view, state kept
  frame   adop_render_forward alone: a viewer's frame, no state kept
  grad    autograd.rasterize and its backward, one or several cameras
  env     a step with a learned environment map, exposure, white balance and
          vignette: forward, backward, adop_env_backward and
          adop_photometric_backward
  photo   camera calibration: forward with a response curve, then
          adop_photometric_backward
  radius  adop_point_radius, the preprocessing of stochastic discarding
  serve   a burst of requests on a Server with two resident clouds

Scenes are surfaces sampled in blocked order (neighbouring indices are
neighbours in space) or the same points in random order:
  spheres  3 spheres, about a unit wide
  room     25 planes and 25 spheres in a 10 m box, seen from 12 m
  site     250 planes and 250 spheres in a 100 m box, seen from 60 m

The discrete part of exact() (which pixel, which depth, who passes the fuzzy
test) follows the FP32 sequence of operations that include/adop.h prescribes;
everything after it is FP64.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2110_06635_gb300 as adop
from paper_2110_06635_gb300 import autograd as adop_autograd

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
BYTES = {"f32": 4, "bf16": 2, "f16": 2}
ALPHA, ZNEAR, GAMMA = 0.01, 1e-3, 1.5
ENV_SIZE = 1024  # the environment map of the paper: 1024 x 1024
LUT = 256
SERVE_SIZES = ((640, 480), (1280, 720), (1920, 1080), (3840, 2160))


def listed():
    return [
        # the smallest call: launches and the host path decide
        dict(name="step_tiny", kind="step", scene="spheres", order="surface", n=20_000, c=4, feat="f32", out="f32",
             w=256, h=256, levels=4),
        # a training crop (512 x 512) of the paper's smallest cloud through autograd, pose and intrinsics too
        dict(name="grad_crop", kind="grad", scene="room", order="surface", n=1_348_406, c=4, feat="bf16", out="bf16",
             w=512, h=512, levels=4, cams=1, keep=True),
        # an unsorted scan with normals, odd sizes, three channels, five layers, gradients summed onto others
        dict(name="step_ragged", kind="step", scene="room", order="random", n=777_773, c=3, feat="f32", out="f32",
             w=1237, h=821, levels=5, normals=True, assign=False, background=True),
        # one full-HD view with FP32 descriptors, points in random order
        dict(name="step_hd_f32_random", kind="step", scene="room", order="random", n=2_570_810, c=8, feat="f32",
             out="f32", w=1920, h=1080, levels=4),
        # the benchmark's view: 5M points, full HD, BF16
        dict(name="step_hd_bf16", kind="step", scene="room", order="surface", n=5_000_000, c=8, feat="bf16",
             out="bf16", w=1920, h=1080, levels=4),
        # the same with stochastic point discarding, FP16, 16-bit gradients in and out
        dict(name="step_discard_f16", kind="step", scene="room", order="surface", n=5_000_000, c=8, feat="f16",
             out="f16", w=1920, h=1080, levels=4, discard=True, grad="f16", gfeat="f16"),
        # a view whose empty pixels show a learned environment map, with learned exposure, white balance and vignette
        dict(name="env_hd_f32", kind="env", scene="room", order="surface", n=2_570_810, c=4, feat="f32", out="f32",
             w=1920, h=1080, levels=4),
        # a training step of twelve mixed views of 20M points, re-rendered in the backward pass
        dict(name="grad_12cam", kind="grad", scene="room", order="surface", n=20_000_000, c=8, feat="bf16",
             out="bf16", w=1920, h=1080, levels=4, cams=12, keep=False),
        # a 4K frame of a 120M-point site in a viewer
        dict(name="frame_4k_120M", kind="frame", scene="site", order="surface", n=120_000_000, c=4, feat="f16",
             out="f16", w=3840, h=2160, levels=4),
        # forward + backward of that cloud at full HD
        dict(name="step_hd_120M", kind="step", scene="site", order="surface", n=120_000_000, c=4, feat="bf16",
             out="bf16", w=1920, h=1080, levels=4),
        # distances to the fourth neighbour of a whole cloud
        dict(name="radius_5M", kind="radius", scene="room", order="surface", n=5_000_000),
        # sixteen requests of mixed sizes that reach a server at once, two clouds resident
        dict(name="serve_16", kind="serve", scene="room", order="surface", n=8_000_000, c=8, feat="bf16", out="bf16",
             w=0, h=0, levels=4, requests=16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 5 + ["frame"] * 2 + ["grad"] * 2 + ["env", "photo", "radius", "serve"])
    scene = rng.choice(["room", "room", "room", "site", "spheres"])
    case = dict(kind=kind, scene=scene, order=rng.choice(["surface", "surface", "surface", "random"]))
    if kind == "radius":
        return dict(case, n=_log_int(rng, 10_000, 5_000_000))
    c = rng.choice([1, 2, 3, 4, 4, 8, 8, 8, 16])
    feat = rng.choice(["f32", "bf16", "bf16", "f16"])
    w = _log_int(rng, 192, 3000)
    case.update(c=c, feat=feat, out=rng.choice(["f32", feat]), w=w, h=max(96, int(w * rng.uniform(0.5, 1.0))),
                levels=rng.choice([1, 3, 4, 4, 4, 4, 5]))
    big = 60_000_000 if kind in ("step", "frame") and c <= 8 else 8_000_000
    case["n"] = _log_int(rng, 5_000, big)
    if kind == "grad":
        case.update(cams=rng.choice([1, 1, 2, 5]), keep=rng.random() < 0.5)
    if kind == "step":
        grad = rng.choice(["f32", "f32", "f32", feat])
        case.update(discard=rng.random() < 0.2, normals=rng.random() < 0.2, log=rng.random() < 0.2,
                    fisheye=rng.random() < 0.2, background=rng.random() < 0.3, grad=grad)
        if rng.random() < 0.3:
            case["assign"] = False
        else:
            case["gfeat"] = grad
    if kind == "serve":
        case.update(order="surface", scene="room", out=feat, requests=rng.randint(4, 20), n=_log_int(rng, 100_000, 8_000_000))
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _surfaces(scene):
    """The scene's surfaces, the same for every seed (the layout decides how much work a view is)."""
    rng = np.random.default_rng({"spheres": 11, "room": 12, "site": 13}[scene])
    out = []
    if scene == "spheres":
        for r in (0.25, 0.35, 0.45):
            out.append(("sphere", rng.uniform(-0.5, 0.5, 3), r, r * r * 4 * math.pi))
        return out
    count, box = (25, 10.0) if scene == "room" else (250, 100.0)
    scale = 2.5 * box / 10.0
    for _ in range(count):
        a, b = rng.uniform(1.0, 6.0, 2) * scale
        q, _ = np.linalg.qr(rng.normal(size=(3, 3)))
        out.append(("plane", rng.uniform(-box / 2, box / 2, 3), (a, b, q), a * b))
    for _ in range(count):
        r = rng.uniform(0.3, 2.0) * scale
        out.append(("sphere", rng.uniform(-box / 2, box / 2, 3), r, r * r * 4 * math.pi))
    return out


def _cloud(case, gen, n=None):
    """xyz, normals (n x 3 float32) of points on the scene's surfaces."""
    n = n or case["n"]
    surf = _surfaces(case["scene"])
    area = np.array([s[3] for s in surf])
    share = np.floor(n * np.cumsum(area) / area.sum() + 0.5).astype(np.int64)
    share[-1] = n
    counts = np.diff(np.concatenate([[0], share]))
    dev = "cuda"
    xyz = torch.empty((n, 3), dtype=torch.float32, device=dev)
    nrm = torch.empty((n, 3), dtype=torch.float32, device=dev) if case.get("normals") else None
    o = 0
    for (shape, centre, size, _), m in zip(surf, (int(v) for v in counts)):
        if m == 0:
            continue
        aspect = 2.0 if shape == "sphere" else size[0] / size[1]
        gx = 8 * max(1, round(math.sqrt(m * aspect) / 8))
        gy = 8 * -(-m // (8 * gx))
        j = torch.arange(m, device=dev) * (gx * gy) // m  # cells in 8 x 8 blocks
        b, r = j // 64, j % 64
        jit = torch.rand((2, m), generator=gen, device=dev)
        s = ((b % (gx // 8)) * 8 + r % 8 + jit[0]) / gx
        t = ((b // (gx // 8)) * 8 + r // 8 + jit[1]) / gy
        ctr = torch.tensor(centre, dtype=torch.float32, device=dev)
        if shape == "sphere":
            z = 2 * t - 1
            rr = torch.sqrt(torch.clamp(1 - z * z, min=0))
            d = torch.stack([rr * torch.cos(2 * math.pi * s), rr * torch.sin(2 * math.pi * s), z], 1)
            xyz[o:o + m] = ctr + size * d
            if nrm is not None:
                nrm[o:o + m] = d
        else:
            a, bb, q = size
            qt = torch.tensor(q, dtype=torch.float32, device=dev)
            xyz[o:o + m] = ctr + ((s - 0.5) * a)[:, None] * qt[:, 0] + ((t - 0.5) * bb)[:, None] * qt[:, 1]
            if nrm is not None:
                nrm[o:o + m] = qt[:, 2]
        o += m
    xyz += 1e-3 * torch.randn((n, 3), generator=gen, device=dev)
    if case["order"] == "random":
        p = torch.randperm(n, generator=gen, device=dev)
        xyz = xyz[p]
        nrm = None if nrm is None else nrm[p]
    return xyz.contiguous(), None if nrm is None else nrm.contiguous()


def _camera(case, rng, k=0, of=1, w=None, h=None):
    """Camera k of `of` on an orbit around the scene, jittered by the seed."""
    w, h = w or case["w"], h or case["h"]
    radius = {"spheres": 2.0, "room": 12.0, "site": 60.0}[case["scene"]]
    az = 0.9 + 2 * math.pi * k / of + rng.normal(scale=0.01)
    el = 0.2 * math.sin(1.0 + 2.0 * k) + rng.normal(scale=0.01)
    eye = radius * np.array([math.cos(el) * math.cos(az), math.sin(el), math.cos(el) * math.sin(az)])
    f = -eye + rng.normal(scale=0.02 * radius, size=3)
    f /= np.linalg.norm(f)
    x = np.cross(f, [0.0, -1.0, 0.0])
    x /= np.linalg.norm(x)
    R = np.stack([x, np.cross(f, x), f])
    cam = SimpleNamespace(w=w, h=h, fx=float(np.float32(0.78 * max(w, h))), fy=float(np.float32(0.78 * max(w, h))),
                          cx=w / 2, cy=h / 2, k1=float(np.float32(-0.05)), k2=float(np.float32(0.01)), k3=0.0, p1=0.0,
                          p2=0.0, model=1 if case.get("fisheye") else 0, R=R.astype(np.float32),
                          t=(-R @ eye).astype(np.float32), epilogue=False, ev=0.0, wb=(1.0, 1.0, 1.0),
                          vig_c=(0.5, 0.5), vig_a=(0.0, 0.0, 0.0))
    if case["kind"] in ("env", "photo", "serve") or (case["kind"] == "grad" and case["cams"] > 1):
        cam.epilogue = True
        cam.ev = float(np.float32(rng.uniform(-1, 1)))
        cam.wb = (float(np.float32(rng.uniform(0.8, 1.2))), 1.0, float(np.float32(rng.uniform(0.8, 1.2))))
        cam.vig_a = (float(np.float32(-0.1)), 0.0, 0.0)
    return cam


def _inputs(case, seed):
    """Everything that is drawn: a namespace of tensors and cameras."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    rng = np.random.default_rng(seed)
    i = SimpleNamespace(normals=None, radius=None, beta=None, env=None, lut=None, background=None, grads=None)
    i.xyz, i.normals = _cloud(case, gen)
    if case["kind"] == "radius":
        return i
    n, c, levels = case["n"], case["c"], case["levels"]

    def descriptors(count):
        f = torch.randn((count, c), generator=gen, device="cuda")
        if case["kind"] in ("photo", "serve"):
            f = torch.exp(0.5 * f - 1.0)  # radiance, under a response curve on [0, 1]
        elif case.get("log"):
            f = 0.5 * f
        return f.to(DTYPES[case["feat"]])

    i.feat = descriptors(n)
    if case["kind"] == "serve":  # the second resident cloud is an eighth of the first
        small = dict(case, scene="spheres")
        i.xyz2, _ = _cloud(small, gen, max(1000, n // 8))
        i.feat2 = descriptors(max(1000, n // 8))
        i.lut = _lut()
        i.requests = []
        for k in range(case["requests"]):
            w, h = SERVE_SIZES[k % 4]
            which = int(k % 3 == 2)
            i.requests.append((which, _camera(small if which else case, rng, k, case["requests"], w, h)))
        return i
    cams = case.get("cams", 1)
    sizes = [(case["w"] * s // 4, case["h"] * s // 4) for s in ((4,) if cams == 1 else (2, 3, 4))]
    i.cams = [_camera(case, rng, k, cams, *sizes[k % len(sizes)]) for k in range(cams)]
    if case.get("background"):
        i.background = torch.randn(c, generator=gen, device="cuda")
    if case.get("discard"):
        # the spacing of the points is what a radius preprocess would find, about
        area = sum(s[3] for s in _surfaces(case["scene"]))
        i.radius = (1.1 * math.sqrt(area / n)) * (0.8 + 0.4 * torch.rand(n, generator=gen, device="cuda"))
        i.beta = torch.rand(n, generator=gen, device="cuda")
    if case["kind"] == "env":
        i.env = 0.5 + 0.3 * torch.randn((ENV_SIZE, ENV_SIZE, c), generator=gen, device="cuda")
    if case["kind"] == "photo":
        i.lut = _lut()
    if case["kind"] != "frame":
        dt = DTYPES[case["out"] if case["kind"] == "grad" else case.get("grad", "f32")]
        lv = 1 if case["kind"] == "photo" else levels
        i.grads = [[torch.randn((c, m.h >> l, m.w >> l), generator=gen, device="cuda").to(dt) for l in range(lv)]
                   for m in i.cams]
    return i


def _lut():
    """The paper's initial response curve x^0.45."""
    x = torch.linspace(0.0, 1.0, LUT, device="cuda")
    return torch.stack([x ** 0.45] * 3).contiguous()


def _flags(case):
    f = 0
    f |= adop.ADOP_FLAG_NORMAL_CULL if case.get("normals") else 0
    f |= adop.ADOP_FLAG_DISCARD if case.get("discard") else 0
    f |= adop.ADOP_FLAG_LOG_DESCRIPTORS if case.get("log") else 0
    f |= adop.ADOP_FLAG_GRAD_ASSIGN if case.get("assign", True) and case["kind"] in ("step", "env") else 0
    f |= adop.ADOP_FLAG_EPILOGUE if case["kind"] in ("env", "photo") or case.get("cams", 1) > 1 else 0
    f |= adop.ADOP_FLAG_LEAKY_CRF if case["kind"] == "photo" else 0
    return f


def prepare(case, seed):
    i = _inputs(case, seed)
    s = SimpleNamespace(case=case, i=i)
    if case["kind"] == "radius":
        return s
    n, c, levels, out = case["n"], case["c"], case["levels"], DTYPES[case["out"]]
    if case["kind"] == "grad":
        s.xyz, s.feat = i.xyz.requires_grad_(), i.feat.requires_grad_()
        s.xi = torch.zeros((len(i.cams), 6), device="cuda", requires_grad=True)
        s.intr = torch.tensor([[m.fx, m.fy, m.cx, m.cy, m.k1, m.k2] for m in i.cams], device="cuda",
                              requires_grad=True)
        return s
    if case["kind"] == "serve":
        s.server = adop.Server(6 << 30, max_slots=64, streams=4, max_batch=8, levels=levels, alpha=ALPHA, znear=ZNEAR,
                               flags=adop.ADOP_FLAG_EPILOGUE, out_dtype=out)
        s.clouds = [s.server.load_cloud(adop.Points(i.xyz, i.feat)), s.server.load_cloud(adop.Points(i.xyz2, i.feat2))]
        s.outs = [torch.empty(adop.output_numel(m, c, levels), dtype=out, device="cuda") for _, m in i.requests]
        torch.cuda.synchronize()  # the server renders on its own streams
        return s
    s.points = adop.Points(i.xyz, i.feat, i.normals, i.radius, i.beta)
    s.params = adop.Params(levels, ALPHA, ZNEAR, i.background, _flags(case), GAMMA, i.env)
    s.luts = None if i.lut is None else [i.lut]
    keep = case["kind"] != "frame"
    s.frames = [adop.Frame.alloc(m, c, levels, out, keep, "cuda", n if keep and case["kind"] != "photo" else None)
                for m in i.cams]
    s.ws = adop.alloc_workspace(s.points, i.cams, s.params, s.luts)
    if case["kind"] in ("step", "env"):
        s.gfeat = torch.zeros((n, c), dtype=DTYPES[case.get("gfeat", "f32")], device="cuda")
        s.gxyz = torch.zeros((n, 3), device="cuda")
        s.gpose, s.gintr = torch.zeros((1, 6), device="cuda"), torch.zeros((1, 6), device="cuda")
    if case["kind"] == "env":
        s.genv = torch.zeros_like(i.env)
    if case["kind"] in ("env", "photo"):
        s.gphoto = torch.zeros((1, 9), device="cuda")
        s.gcrf = None if i.lut is None else torch.zeros_like(i.lut)
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(s):
    case, i = s.case, s.i
    kind = case["kind"]
    if kind == "radius":
        return adop.adop_point_radius(i.xyz)
    if kind == "grad":
        images = adop_autograd.rasterize(s.xyz, s.feat, i.cams, s.xi, s.intr, levels=case["levels"], alpha=ALPHA,
                                         znear=ZNEAR, flags=_flags(case), out_dtype=DTYPES[case["out"]],
                                         keep_state=case["keep"])
        flat = [im for per in images for im in per]
        g = torch.autograd.grad(flat, [s.xyz, s.feat, s.xi, s.intr], [g for per in i.grads for g in per])
        return {"images": [im.detach() for im in flat], "grads": list(g)}
    if kind == "serve":
        tickets = [s.server.submit(s.clouds[which], m, out, i.lut) for (which, m), out in zip(i.requests, s.outs)]
        for t in tickets:
            if s.server.wait(t) != 0:
                raise RuntimeError("a request did not finish")
        return s.outs
    adop.adop_render_forward(s.points, i.cams, s.params, s.frames, s.ws, crf_luts=s.luts)
    fr = s.frames[0]
    if kind == "frame":
        return fr.images
    if kind == "photo":
        s.gphoto.zero_()
        s.gcrf.zero_()
        adop.adop_photometric_backward(i.cams, s.params, case["c"], s.frames, [i.grads[0][0]], s.gphoto, s.gcrf,
                                       crf_luts=s.luts)
        return {"images": fr.images, "key": fr.key, "count": fr.count, "grads": [s.gphoto, s.gcrf]}
    if not case.get("assign", True):
        s.gfeat.zero_()
        s.gxyz.zero_()
    s.gpose.zero_()
    s.gintr.zero_()
    adop.adop_render_backward(s.points, i.cams, s.params, s.frames, i.grads, s.gfeat, s.gxyz, s.gpose, s.gintr, s.ws,
                              crf_luts=s.luts)
    grads = [s.gxyz, s.gfeat, s.gpose, s.gintr]
    if kind == "env":
        s.genv.zero_()
        adop.adop_env_backward(i.cams, s.params, case["c"], s.frames, i.grads, s.genv, crf_luts=s.luts)
        s.gphoto.zero_()
        adop.adop_photometric_backward(i.cams, s.params, case["c"], s.frames, [i.grads[0][0]], s.gphoto)
        grads += [s.genv, s.gphoto]
    return {"images": fr.images, "key": fr.key, "count": fr.count, "grads": grads}


def _pixels(w, h, levels):
    return sum((w >> l) * (h >> l) for l in range(levels))


def work(case):
    """Inputs read once (positions, descriptors, upstream gradients, map),
    outputs written once (images, kept keys and counts, gradients)."""
    n, kind = case["n"], case["kind"]
    if kind == "radius":
        return {"bytes": 16.0 * n, "flops": 9.0 * 32 * n}  # a neighbourhood's candidates
    c, levels = case["c"], case["levels"]
    point = 12 + c * BYTES[case["feat"]]
    out = c * BYTES[case["out"]]
    if kind == "serve":
        px = sum(_pixels(*SERVE_SIZES[k % 4], levels) for k in range(case["requests"]))
        views = sum(n // 8 if k % 3 == 2 else n for k in range(case["requests"]))
        return {"bytes": float(point * (n + n // 8) + px * out), "flops": 60.0 * views}
    if kind == "frame":
        return {"bytes": float(n * point + _pixels(case["w"], case["h"], levels) * out), "flops": 60.0 * n}
    if kind == "photo":
        px = _pixels(case["w"], case["h"], levels)
        return {"bytes": float(n * point + px * (out + 12) + 4 * c * case["w"] * case["h"]), "flops": 60.0 * n}
    if kind == "grad":
        cams = case["cams"]
        scales = (4,) if cams == 1 else (2, 3, 4)
        px = sum(_pixels(case["w"] * s // 4, case["h"] * s // 4, levels)
                 for s in (scales[k % len(scales)] for k in range(cams)))
        return {"bytes": float(n * (2 * point) + px * 2 * out), "flops": 120.0 * n * cams}
    px = _pixels(case["w"], case["h"], levels)
    normals = 12 if case.get("normals") else 0
    discard = 8 if case.get("discard") else 0
    env = 8 * ENV_SIZE * ENV_SIZE * c if kind == "env" else 0
    return {"bytes": float(n * (point + normals + discard + 12 + c * BYTES[case.get("gfeat", "f32")])
                           + px * (out + 12 + c * BYTES[case.get("grad", "f32")]) + env), "flops": 120.0 * n}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

CHUNK = 4_000_000
F32 = np.float32
D = torch.float64


def _project(cam, x, nrm=None):
    """u0, v0, depth (float32, one rounding per operation) and who is valid."""
    R, t = [float(v) for v in np.asarray(cam.R, F32).ravel()], [float(v) for v in np.asarray(cam.t, F32)]
    X = [((R[3 * r] * x[:, 0] + R[3 * r + 1] * x[:, 1]) + R[3 * r + 2] * x[:, 2]) + t[r] for r in range(3)]
    one = torch.ones((), device=x.device)
    if cam.model == 1:
        z = torch.sqrt((X[0] * X[0] + X[1] * X[1]) + X[2] * X[2])
        s = z + X[2]
        ok = s > 0
        a = (2.0 * one) / s
        xn, yn = a * X[0], a * X[1]
    else:
        z, ok = X[2], torch.ones_like(X[2], dtype=torch.bool)
        xn, yn = X[0] / z, X[1] / z
    r2 = xn * xn + yn * yn
    d = r2 * (cam.k1 + r2 * (cam.k2 + r2 * cam.k3)) + 1.0
    u0, v0 = cam.fx * (xn * d) + cam.cx, cam.fy * (yn * d) + cam.cy
    ok = ok & (z > F32(ZNEAR).item())
    if nrm is not None:
        q = [(R[3 * r] * nrm[:, 0] + R[3 * r + 1] * nrm[:, 1]) + R[3 * r + 2] * nrm[:, 2] for r in range(3)]
        ok = ok & (((q[0] * X[0] + q[1] * X[1]) + q[2] * X[2]) > 0)
    return u0, v0, z, ok


def _pixel(cam, u0, v0, l):
    """Pixel coordinates at layer l and who is inside."""
    ul, vl = u0 * 2.0 ** -l, v0 * 2.0 ** -l
    w, h = cam.w >> l, cam.h >> l
    ok = (ul > -1) & (ul < w + 1) & (vl > -1) & (vl < h + 1)
    pu = torch.round(torch.where(ok, ul, -1.0 * torch.ones_like(ul))).long()
    pv = torch.round(torch.where(ok, vl, -1.0 * torch.ones_like(vl))).long()
    return pu, pv, ok & (pu >= 0) & (pu < w) & (pv >= 0) & (pv < h)


def _taps(cam, l, ew, eh):
    """Texel indices and weights (4 x pixels) of layer l's rays (radial lenses)."""
    w, h = cam.w >> l, cam.h >> l
    v, u = torch.meshgrid(torch.arange(h, device="cuda", dtype=D), torch.arange(w, device="cuda", dtype=D),
                          indexing="ij")
    xd, yd = (u.ravel() * 2 ** l - cam.cx) / cam.fx, (v.ravel() * 2 ** l - cam.cy) / cam.fy
    rd = torch.sqrt(xd * xd + yd * yd)
    r = rd.clone()
    for _ in range(30):
        q = r * r
        f = r * (1 + q * (cam.k1 + q * (cam.k2 + q * cam.k3))) - rd
        r = r - f / (1 + q * (3 * cam.k1 + q * (5 * cam.k2 + q * 7 * cam.k3)))
    s = torch.where(rd > 0, r / torch.clamp(rd, min=1e-300), torch.ones_like(rd))
    d = torch.stack([xd * s, yd * s, torch.ones_like(xd)], 1)
    d = d / d.norm(dim=1, keepdim=True)
    d = d @ torch.tensor(np.asarray(cam.R, np.float64), device="cuda")  # R^T d
    ue = (torch.atan2(d[:, 0], d[:, 2]) + math.pi) * ew / (2 * math.pi) - 0.5
    ve = torch.acos(torch.clamp(d[:, 1], -1, 1)) * eh / math.pi - 0.5
    iu, iv = torch.floor(ue), torch.floor(ve)
    fu, fv = ue - iu, ve - iv
    ua = iu.long() % ew
    ub = (ua + 1) % ew
    va, vb = iv.long().clamp(0, eh - 1), (iv.long() + 1).clamp(0, eh - 1)
    t = torch.stack([va * ew + ua, va * ew + ub, vb * ew + ua, vb * ew + ub])
    return t, torch.stack([(1 - fu) * (1 - fv), fu * (1 - fv), (1 - fu) * fv, fu * fv])


def _photometric(cam, lut, leaky, I):
    """The photometric model on layer 0 (pixels x c): output, d out / d in, and
    what the parameter gradients need."""
    h, w = cam.h, cam.w
    v, u = torch.meshgrid(torch.arange(h, device="cuda", dtype=D), torch.arange(w, device="cuda", dtype=D),
                          indexing="ij")
    ru, rv = u.ravel() / w - cam.vig_c[0], v.ravel() / h - cam.vig_c[1]
    r2 = ru * ru + rv * rv
    a = cam.vig_a
    vig = 1 + r2 * (a[0] + r2 * (a[1] + r2 * a[2]))
    out, slope = I.clone(), torch.ones_like(I)
    parts = []
    for ch in range(min(3, I.shape[1])):
        scale = 2.0 ** -cam.ev * cam.wb[ch] * vig
        x = I[:, ch] * scale
        y, sl, seg, fr = x, torch.ones_like(x), None, None
        if lut is not None:
            n = lut.shape[1]
            pos = x.clamp(0, 1) * (n - 1)
            seg = torch.floor(pos).long().clamp(max=n - 2)
            fr = pos - seg
            lo, hi = lut[ch].to(D)[seg], lut[ch].to(D)[seg + 1]
            y, sl = lo * (1 - fr) + hi * fr, (hi - lo) * (n - 1)
            if leaky:
                up, dn = x > 1, x < 0
                q = torch.where(up, x, torch.ones_like(x))
                y = torch.where(up, -0.01 / torch.sqrt(q) + 1.01, torch.where(dn, 0.01 * x, y))
                sl = torch.where(up, 0.005 * q ** -1.5, torch.where(dn, 0.01 * torch.ones_like(x), sl))
                fr = torch.where(up | dn, torch.full_like(fr, float("nan")), fr)
            else:
                sl = torch.where((x < 0) | (x > 1), torch.zeros_like(sl), sl)
        out[:, ch], slope[:, ch] = y, sl * scale
        parts.append((x, sl, seg, fr))
    return out, slope, (ru, rv, r2, vig, parts)


def _render(case, i, cam, xyz, feat, normals):
    """Per layer: key, count, blended value before the photometric model."""
    n, c, levels = xyz.shape[0], feat.shape[1], case["levels"]
    sizes = [(cam.w >> l) * (cam.h >> l) for l in range(levels)]
    big = torch.iinfo(torch.int64).max
    keys = [torch.full((m,), big, dtype=torch.int64, device="cuda") for m in sizes]
    a1 = float(F32(1.0) + F32(ALPHA))

    def pairs():
        for o in range(0, n, CHUNK):
            e = min(n, o + CHUNK)
            u0, v0, z, ok = _project(cam, xyz[o:e], None if normals is None else normals[o:e])
            for l in range(levels):
                pu, pv, inside = _pixel(cam, u0, v0, l)
                inside = inside & ok
                if i.radius is not None:
                    t = (float(F32(cam.fx) * F32(2.0 ** -l)) * i.radius[o:e]) / z
                    inside = inside & ((t * t) * float(F32(GAMMA) * F32(GAMMA)) > 1.0 - i.beta[o:e])
                j = inside.nonzero().ravel()
                yield l, j + o, (pv * (cam.w >> l) + pu)[j], z[j], pu[j], pv[j]

    for l, j, p, z, _, _ in pairs():
        keys[l].scatter_reduce_(0, p, (z.view(torch.int32).long() << 32) | j, "amin")
    zmin = [torch.where(k == big, float("inf"), (k >> 32).int().view(torch.float32)) for k in keys]
    cnt = [torch.zeros(m, dtype=D, device="cuda") for m in sizes]
    acc = [torch.zeros((m, c), dtype=D, device="cuda") for m in sizes]
    member = [[] for _ in range(levels)]
    for l, j, p, z, pu, pv in pairs():
        q = (z <= zmin[l][p] * a1).nonzero().ravel()
        j, p = j[q], p[q]
        tau = feat[j].to(D)
        tau = torch.exp(tau) if case.get("log") else tau
        cnt[l].index_add_(0, p, torch.ones(p.numel(), dtype=D, device="cuda"))
        acc[l].index_add_(0, p, tau)
        member[l].append((j, z[q], pu[q], pv[q]))
    I = []
    for l in range(levels):
        v = acc[l] / cnt[l].clamp(min=1)[:, None]
        e = cnt[l] == 0
        if i.env is not None:
            t, w = _taps(cam, l, i.env.shape[1], i.env.shape[0])
            flat = i.env.reshape(-1, c).to(D)
            v[e] = sum(w[k][e, None] * flat[t[k][e]] for k in range(4))
        elif i.background is not None:
            v[e] = i.background.to(D)
        I.append(v)
    return keys, cnt, zmin, I, [tuple(torch.cat(x) for x in zip(*m)) if m else None for m in member]


def _chain(cam, xyz, du, dv):
    """dL/dX, the intrinsics terms, and X (camera space)."""
    R = torch.tensor(np.asarray(cam.R, np.float64), device="cuda")
    X = xyz.to(D) @ R.T + torch.tensor(np.asarray(cam.t, np.float64), device="cuda")
    gxd, gyd = cam.fx * du, cam.fy * dv
    if cam.model == 1:
        d = X.norm(dim=1)
        s = d + X[:, 2]
        a = 2 / s
        xn, yn = a * X[:, 0], a * X[:, 1]
    else:
        xn, yn = X[:, 0] / X[:, 2], X[:, 1] / X[:, 2]
    r2 = xn * xn + yn * yn
    rad = 1 + r2 * (cam.k1 + r2 * (cam.k2 + r2 * cam.k3))
    drad = cam.k1 + r2 * (2 * cam.k2 + 3 * cam.k3 * r2)
    gxn = gxd * (rad + 2 * xn * xn * drad) + gyd * 2 * xn * yn * drad
    gyn = gxd * 2 * xn * yn * drad + gyd * (rad + 2 * yn * yn * drad)
    if cam.model == 1:
        q = -2 / (s * s) * (gxn * X[:, 0] + gyn * X[:, 1])
        dX = torch.stack([gxn * a + q * X[:, 0] / d, gyn * a + q * X[:, 1] / d, q * (X[:, 2] / d + 1)], 1)
    else:
        dX = torch.stack([gxn, gyn, -(gxn * xn + gyn * yn)], 1) / X[:, 2:3]
    terms = [du * xn * rad, dv * yn * rad, du, dv, (gxd * xn + gyd * yn) * r2, (gxd * xn + gyd * yn) * r2 * r2]
    pose = torch.cat([dX.sum(0), torch.linalg.cross(X, dX).sum(0)])
    return dX @ R, pose, torch.stack([t.sum() for t in terms])


def _backward(case, cam, xyz, feat, G, cnt, zmin, I, member, gxyz, gfeat):
    """Adds one camera's gradients to gxyz and gfeat; returns pose and intrinsics."""
    n = xyz.shape[0]
    a1 = float(F32(1.0) + F32(ALPHA))
    du, dv = torch.zeros(n, dtype=D, device="cuda"), torch.zeros(n, dtype=D, device="cuda")
    for l, m in enumerate(member):
        if m is None:
            continue
        w, h = cam.w >> l, cam.h >> l
        for o in range(0, m[0].numel(), CHUNK):
            j, z, pu, pv = (x[o:o + CHUNK] for x in m)
            p = pv * w + pu
            tau = feat[j].to(D)
            tau = torch.exp(tau) if case.get("log") else tau
            gf = G[l][p] / cnt[l][p, None]
            gfeat.index_add_(0, j, gf * tau if case.get("log") else gf)
            side = []
            for su, sv in ((1, 0), (-1, 0), (0, 1), (0, -1)):
                qu, qv = pu + su, pv + sv
                inside = (qu >= 0) & (qu < w) & (qv >= 0) & (qv < h)
                q = torch.where(inside, qv * w + qu, torch.zeros_like(p))
                zq, nq = zmin[l][q], cnt[l][q]
                wgt = 1 / (1 + nq)
                wgt = torch.where(z * a1 < zq, torch.ones_like(wgt), wgt)
                wgt = torch.where(z > zq * a1, torch.zeros_like(wgt), wgt)
                wgt = torch.where(nq == 0, torch.ones_like(wgt), wgt) * inside
                side.append(wgt * (G[l][q] * (tau - I[l][q])).sum(1))
            du.index_add_(0, j, 0.5 * (side[0] - side[1]) * 2.0 ** -l)
            dv.index_add_(0, j, 0.5 * (side[2] - side[3]) * 2.0 ** -l)
    pose, intr = torch.zeros(6, dtype=D, device="cuda"), torch.zeros(6, dtype=D, device="cuda")
    hit = ((du != 0) | (dv != 0)).nonzero().ravel()
    for o in range(0, hit.numel(), CHUNK):
        j = hit[o:o + CHUNK]
        gx, p, q = _chain(cam, xyz[j], du[j], dv[j])
        gxyz.index_add_(0, j, gx)
        pose += p
        intr += q
    return pose, intr


def _planar(v, cam, l):
    return v.T.reshape(v.shape[1], cam.h >> l, cam.w >> l)


def exact(case, seed):
    if case["kind"] == "radius":
        return None  # an exhaustive search of a whole cloud takes too long
    i = _inputs(case, seed)
    kind, levels = case["kind"], case["levels"]
    if kind == "serve":
        outs = []
        for which, cam in i.requests:
            _, _, _, I, _ = _render(case, i, cam, i.xyz2 if which else i.xyz, i.feat2 if which else i.feat, None)
            I[0] = _photometric(cam, i.lut, False, I[0])[0]
            outs.append(torch.cat([v.T.reshape(-1) for v in I]))
        return outs
    images, gxyz, gfeat, poses, intrs = [], None, None, [], []
    if kind not in ("frame", "photo"):
        gxyz = torch.zeros((case["n"], 3), dtype=D, device="cuda")
        gfeat = torch.zeros((case["n"], case["c"]), dtype=D, device="cuda")
    for k, cam in enumerate(i.cams):
        keys, cnt, zmin, I, member = _render(case, i, cam, i.xyz, i.feat, i.normals)
        shown, slope = list(I), None
        if cam.epilogue:
            shown[0], slope, photo = _photometric(cam, i.lut, kind == "photo", I[0])
        images += [_planar(v, cam, l) for l, v in enumerate(shown)]
        if kind == "frame":
            return images
        G = [g.to(D).reshape(case["c"], -1).T.contiguous() for g in i.grads[k]]
        if kind == "photo":
            return {"images": images, "key": None, "count": None, "grads": _photo_grads(cam, i.lut, G[0], I[0], photo)}
        if kind == "env":
            gphoto = _photo_grads(cam, None, G[0], I[0], photo)
        if slope is not None:
            G[0] = G[0] * slope
        p, q = _backward(case, cam, i.xyz, i.feat, G, cnt, zmin, I, member, gxyz, gfeat)
        poses.append(p)
        intrs.append(q)
        if kind == "env":
            genv = torch.zeros((ENV_SIZE * ENV_SIZE, case["c"]), dtype=D, device="cuda")
            for l in range(levels):
                e = (cnt[l] == 0).nonzero().ravel()
                t, w = _taps(cam, l, ENV_SIZE, ENV_SIZE)
                for s in range(4):
                    genv.index_add_(0, t[s][e], w[s][e, None] * G[l][e])
    grads = [gxyz, gfeat, torch.stack(poses), torch.stack(intrs)]
    if kind == "grad":
        return {"images": images, "grads": grads}
    if kind == "env":
        grads += [genv.view(ENV_SIZE, ENV_SIZE, case["c"]), gphoto[0]]
    return {"images": images, "key": None, "count": None, "grads": grads}


def _photo_grads(cam, lut, G, I, photo):
    """[ev, wb (3), vig_c (2), vig_a (3)] and the response curve's gradient."""
    ru, rv, r2, vig, parts = photo
    a, e = cam.vig_a, 2.0 ** -cam.ev
    dvig = a[0] + r2 * (2 * a[1] + 3 * r2 * a[2])
    out = torch.zeros(9, dtype=D, device="cuda")
    crf = None if lut is None else torch.zeros(lut.shape, dtype=D, device="cuda")
    for ch, (x, sl, seg, fr) in enumerate(parts):
        g = G[:, ch]
        base = g * sl * I[:, ch] * e
        out[0] += (g * sl * x).sum() * -math.log(2)
        out[1 + ch] += (base * vig).sum()
        b = base * cam.wb[ch]
        out[4] += (b * dvig * -2 * ru).sum()
        out[5] += (b * dvig * -2 * rv).sum()
        for k in range(3):
            out[6 + k] += (b * r2 ** (k + 1)).sum()
        if lut is None:
            continue
        on = torch.isfinite(fr).nonzero().ravel()
        crf[ch].index_add_(0, seg[on], (g * (1 - fr))[on])
        crf[ch].index_add_(0, seg[on] + 1, (g * fr)[on])
    return [out[None], crf]
