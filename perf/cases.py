"""Workloads of the Weighted Sum Rendering library, by use, with their FP64 results.

A case is a dict of plain values whose ``path`` names what a program does with the library:

* ``frame``   a viewer's frame: project, bin and render a scene (``Renderer.forward``);
* ``grad``    an image and its gradients in a PyTorch program (``render`` under autograd);
* ``step``    a captured forward + L1 loss + backward (``GraphStep``);
* ``train``   a captured optimisation step, the 3DGS loss and Adam included (``TrainStep``);
* ``chain``   the per-Gaussian layer alone, forward and backward (``wsr_project``, ``wsr_project_bwd``);
* ``loss``    the training loss and its gradient alone (``wsr_loss_3dgs``);
* ``adam``    the optimiser's update alone (``Adam``).

Scenes are drawn on the GPU like the synthetic scenes of the tests and the benchmark: clustered
centres in a box, log-normal scales, SH colours, sigmoid opacities.  ``exact`` renders and
differentiates the same scenes in float64 with plain torch.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2410_18931_gb300 import Adam, FlatParams, Gaussians, GraphStep, Renderer, TrainStep, render
from paper_2410_18931_gb300 import _abi as A

KINDS = {"dir": 0, "exp": 1, "lc": 2}
ORDER = ("means", "log_scales", "quats", "sh", "opacity", "lc_v", "weight_params")
DC = 2.0 * math.sqrt(math.pi)          # a degree-0 SH coefficient of DC * x contributes x
LR = dict(means=1.6e-6, log_scales=5e-5, quats=1e-5, sh=2.5e-5, opacity=5e-4, lc_v=1e-5, weight_params=1e-5)


# --------------------------------------------------------------------------------------------
# The cases
# --------------------------------------------------------------------------------------------

def _case(path, n=0, views="", *, degree=3, vd=True, weight="lc", reduced=False, tile="16x16", persistent=False,
          chunk=0, deterministic=False, spread="cluster"):
    return dict(path=path, n=n, views=views, degree=degree, vd=vd, weight=weight, reduced=reduced, tile=tile,
                persistent=persistent, chunk=chunk, deterministic=deterministic, spread=spread)


def listed():
    return [
        # the smallest interactive frame: a toy scene in a thumbnail, where launches and host calls are the time
        dict(_case("frame", 1000, "128x128", degree=0, vd=False, weight="exp", spread="box"), name="frame-1k-128"),
        # a mid-sized scene at a mobile viewer's resolution, everything at the library's defaults
        dict(_case("frame", 200_000, "1280x720"), name="frame-200k-720p"),
        # a large scene stored in bf16 / f16, two 4K views in one call: the largest frame
        dict(_case("frame", 6_000_000, "3840x2160,3840x2160", reduced=True, persistent=True), name="frame-6M-2x4k"),
        # a small differentiable render inside a PyTorch program (fitting a thumbnail), plain 3DGS opacities
        dict(_case("grad", 3000, "200x120", degree=1, vd=False, weight="dir", spread="box"), name="grad-3k-200x120"),
        # an object capture of a ragged size fitted in a PyTorch program, library defaults
        dict(_case("grad", 150_000, "979x543", degree=2, weight="exp"), name="grad-150k-979x543"),
        # the benchmark's step: a 1M-Gaussian scene at 1080p, tuned schedule, one graph
        dict(_case("step", 1_000_000, "1920x1080", persistent=True, chunk=512), name="step-1M-1080p"),
        # a batch of uneven views in one captured step, library defaults
        dict(_case("step", 300_000, "640x360,1280x720,1920x1080,640x360,1280x720,801x601", degree=2, vd=False,
                   weight="exp", persistent=True), name="step-300k-6-views"),
        # a whole optimisation step over a 720p view
        dict(_case("train", 200_000, "1280x720", persistent=True, chunk=512), name="train-200k-720p"),
        # the same kind of step when results must repeat bit for bit
        dict(_case("step", 250_000, "1280x720", persistent=True, chunk=512, deterministic=True),
             name="deterministic-250k-720p"),
        # the per-Gaussian layer of the benchmark's scene
        dict(_case("chain", 1_000_000, "1920x1080"), name="chain-1M"),
        # the training loss at 1080p
        dict(_case("loss", 0, "1920x1080"), name="loss-1080p"),
        # the optimiser over the benchmark's scene (75 numbers per Gaussian)
        dict(_case("adam", 1_000_000), name="adam-1M"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo, hi):
    w = _log_int(rng, lo, hi)
    return w, max(16, int(w * rng.choice((0.5625, 0.5625, 0.67, 0.75, 1.0))))


def draw(rng):
    path = rng.choice(("frame", "frame", "grad", "grad", "step", "step", "train", "deterministic", "chain", "loss",
                       "adam"))
    views = [_size(rng, 128, 1920) for _ in range(rng.choice((1, 1, 1, 2, 3)))]
    if path in ("grad", "train"):
        views = views[:1]
    name = ",".join("%dx%d" % v for v in views)
    weight = rng.choice(("lc", "lc", "exp", "dir"))
    degree, vd = rng.choice(((3, True), (3, True), (3, False), (2, True), (1, False), (0, False)))
    n = _log_int(rng, 1000, 1_000_000)
    more = dict(degree=degree, vd=vd, weight=weight, spread="box" if n < 8000 else "cluster",
                tile=rng.choice(("16x16", "16x16", "16x16", "16x8", "32x8", "8x8")))
    if path == "frame":
        return _case("frame", n, name, reduced=rng.random() < 0.25, persistent=rng.random() < 0.5, **more)
    if path == "grad":
        return _case("grad", min(n, 500_000), name, **more)
    if path == "step":
        return _case("step", n, name, persistent=rng.random() < 0.8, chunk=rng.choice((0, 128, 256, 512, 512)), **more)
    if path == "train":
        return _case("train", min(n, 400_000), name, persistent=True, chunk=rng.choice((0, 512)), **more)
    if path == "deterministic":
        # a tile's list is bounded in this mode: keep to the densities that stay within the bound
        more.update(tile=rng.choice(("16x16", "16x8")))
        w, h = _size(rng, 320, 1920)
        return _case("step", min(n, int(0.27 * w * h)), "%dx%d" % (w, h), persistent=True,
                     chunk=rng.choice((0, 512)), deterministic=True, **more)
    if path == "chain":
        return _case("chain", n, name, degree=degree, vd=vd, weight=weight)
    if path == "loss":
        return _case("loss", 0, name)
    return _case("adam", n, degree=degree, vd=vd)


# --------------------------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------------------------

def _cameras(case):
    """One view: in front of the scene.  Several: on a Fibonacci sphere around it.  60 degrees of vertical
    field of view, every number a float32."""
    sizes = [tuple(int(x) for x in v.split("x")) for v in case["views"].split(",")]
    dist = 4.0 if case["spread"] == "box" else 5.0
    cams = []
    for j, (w, h) in enumerate(sizes):
        if len(sizes) == 1:
            pos, up = np.array([0.0, 0.0, -dist]), np.array([0.0, 1.0, 0.0])
        else:
            y = 1.0 - 2.0 * (j + 0.5) / len(sizes)
            r, a = math.sqrt(1.0 - y * y), math.pi * (3.0 - math.sqrt(5.0)) * j
            pos = (dist + 1.0) * np.array([r * math.cos(a), y, r * math.sin(a)])
            up = np.array([0.0, 0.0, 1.0]) if abs(y) > 0.95 else np.array([0.0, 1.0, 0.0])
        fwd = -pos / np.linalg.norm(pos)
        right = np.cross(fwd, up)
        right /= np.linalg.norm(right)
        R = np.stack([right, np.cross(fwd, right), fwd]).astype(np.float32).astype(np.float64)
        f = float(np.float32(0.5 * h / math.tan(math.radians(60.0) * 0.5)))
        cams.append(SimpleNamespace(R=R, T=(-R @ pos).astype(np.float32).astype(np.float64), fx=f, fy=f, cx=0.5 * w,
                                    cy=0.5 * h, width=w, height=h, znear=float(np.float32(0.2))))
    return cams


def _scene(case, seed):
    """The scene's float32 tensors and the six weight parameters.  Under a loss with an L1 term the scene's
    colours are dim (at most about 0.6) and its target is bright (0.7 and up), as when a fit begins."""
    g = torch.Generator("cuda").manual_seed(int(seed))
    n, K = case["n"], (case["degree"] + 1) ** 2
    dim = case["path"] in ("step", "train")

    def normal(*s):
        return torch.randn(*s, device="cuda", generator=g)

    def uniform(*s):
        return torch.rand(*s, device="cuda", generator=g)

    if case["spread"] == "box":
        means, mu, sd = 2.0 * uniform(n, 3) - 1.0, -3.0, 0.5
    else:
        centres = 6.0 * uniform(64, 3) - 3.0
        means = centres[torch.randint(64, (n,), device="cuda", generator=g)] + 0.3 * normal(n, 3)
        mu, sd = -4.0, 0.7
    log_scales = mu + sd * normal(n, 3)
    quats = torch.nn.functional.normalize(normal(n, 4), dim=1)
    sh = (0.02 if dim else 0.2) * normal(n, K, 3)
    sh[:, 0] = DC * ((0.4 * uniform(n, 3) - 0.4) if dim else (uniform(n, 3) - 0.5))
    if case["vd"]:
        opacity = 0.05 * normal(n, K)
        opacity[:, 0] = DC * torch.sigmoid(normal(n))
    else:
        opacity = normal(n)
    lc_v = 0.05 + 0.1 * uniform(n)
    if case["reduced"]:
        log_scales, quats, sh, opacity = log_scales.bfloat16(), quats.bfloat16(), sh.half(), opacity.half()
    sigma, beta = {"dir": (0.0, 0.0), "exp": (0.1, 0.8), "lc": (10.0, 0.0)}[case["weight"]]
    wp = torch.tensor([sigma, beta, 1.0, 0.0, 0.0, 0.0], device="cuda")
    return dict(means=means, log_scales=log_scales, quats=quats, sh=sh, opacity=opacity, lc_v=lc_v, weight_params=wp)


def _gaussians(case, s):
    return Gaussians(s["means"], s["log_scales"], s["quats"], s["sh"], s["opacity"], s["lc_v"], case["degree"],
                     case["vd"])


def _pixels(case):
    return sum(c.width * c.height for c in _cameras(case))


def _image(case, seed, kind):
    """``grad``: a loss's gradient per pixel; ``target``: a bright image; ``photo`` and ``fit``: a smooth image
    with grain and one near it."""
    g = torch.Generator("cuda").manual_seed(int(seed) * 7 + 1)
    P = _pixels(case)
    if kind == "grad":
        return torch.randn(P, 3, device="cuda", generator=g) / (3.0 * P)
    if kind == "target":
        return 0.7 + 0.3 * torch.rand(P, 3, device="cuda", generator=g)
    i = torch.arange(P, device="cuda")[:, None]
    photo = 0.5 + 0.3 * torch.sin(i * torch.tensor([0.011, 0.017, 0.023], device="cuda")) \
        + 0.1 * torch.randn(P, 3, device="cuda", generator=g)
    fit = photo + 0.05 * torch.randn(P, 3, device="cuda", generator=g)
    return (photo if kind == "photo" else fit).clamp(0.0, 1.0)


def _record_grads(case, s, seed):
    """Gradient records as a render backward leaves them: moments in each footprint's own frame."""
    g = torch.Generator("cuda").manual_seed(int(seed) * 7 + 2)
    cams, n = _cameras(case), case["n"]
    out = torch.zeros(len(cams), n, 12, device="cuda")
    with torch.no_grad():
        for v, c in enumerate(cams):
            p = _project64(case, {k: t.double() for k, t in s.items()}, c)
            hx = torch.where(p["seen"], p["a"].clamp(max=1e6).sqrt(), 0.0).float()
            z = 1e-6 * torch.randn(n, 9, device="cuda", generator=g) * p["seen"][:, None]
            z *= torch.stack([torch.ones_like(hx), hx, torch.ones_like(hx), hx, hx * hx] + [torch.ones_like(hx)] * 4, 1)
            out[v, :, :9] = z
    return out.reshape(-1)


def _adam_values(case, flat, opt, seed):
    """Parameters, gradients and moments in the middle of a run."""
    g = torch.Generator("cuda").manual_seed(int(seed))
    flat.data.normal_(generator=g)
    flat.grad_data.normal_(0.0, 1e-4, generator=g)
    opt.exp_avg.normal_(0.0, 3e-5, generator=g)
    opt.exp_avg_sq.normal_(0.0, 1e-4, generator=g).square_()
    opt.state[0] = 700


def _adam(case):
    n, K = case["n"], (case["degree"] + 1) ** 2
    flat = FlatParams(dict(means=(n, 3), log_scales=(n, 3), quats=(n, 4), sh=(n, K, 3),
                           opacity=(n, K) if case["vd"] else (n,), lc_v=(n,), weight_params=(6,)))
    return flat, Adam(flat, case["degree"], case["vd"])


def _renderer(case):
    return Renderer(_cameras(case), tile=tuple(int(x) for x in case["tile"].split("x")),
                    persistent=case["persistent"], chunk=case["chunk"], deterministic=case["deterministic"])


def prepare(case, seed):
    path, st = case["path"], SimpleNamespace(case=case)
    if path == "adam":
        st.flat, st.opt = _adam(case)
        _adam_values(case, st.flat, st.opt, seed)
        return st
    if path == "loss":
        st.r = _renderer(case)
        st.rgb, st.target = _image(case, seed, "fit"), _image(case, seed, "photo")
        st.loss, st.grad = torch.zeros(3, device="cuda"), torch.empty_like(st.rgb)
        return st
    s = _scene(case, seed)
    st.kind, st.w, st.g = KINDS[case["weight"]], s["weight_params"], _gaussians(case, s)
    if path in ("step", "train"):
        target = _image(case, seed, "target")
        how = dict(tile=tuple(int(x) for x in case["tile"].split("x")), persistent=case["persistent"],
                   chunk=case["chunk"], deterministic=case["deterministic"])
    if path == "step":
        st.step = GraphStep(st.g, _cameras(case), st.kind, st.w, target, **how)
        return st
    if path == "train":
        flat = FlatParams({k: tuple(s[k].shape) for k in ORDER})
        for k in ORDER:
            flat.param[k].copy_(s[k])
        # the low rates of the end of a run: the scene stays what it is over many passes
        st.step = TrainStep(flat, case["degree"], case["vd"], _cameras(case), st.kind, target, lr=LR, **how)
        return st
    st.r = _renderer(case)
    if path == "chain":
        st.records = torch.empty(st.r.n_cams * case["n"] * A.WSR_RECORD_FLOATS, device="cuda")
        st.grad_records = _record_grads(case, s, seed)
        st.out = {k: torch.empty(s[k].shape, device="cuda") for k in ORDER[:6]}
        st.grads = A.wsr_grads(*[st.out[k].data_ptr() for k in ORDER[:6]], None)
        return st
    st.frame = st.r.forward(st.g, st.kind, st.w)        # sizes the tile list, as a program's first frame does
    if path == "grad":
        st.frame = None
        st.leaves = [s[k].requires_grad_() for k in ORDER]
        st.grad_rgb = _image(case, seed, "grad")
    return st


def run(st):
    case, path = st.case, st.case["path"]
    if path == "frame":
        f = st.r.forward(st.g, st.kind, st.w, st.frame)
        return dict(rgb=f.rgb, den=f.den)
    if path == "grad":
        rgb = render(st.r, st.kind, st.g, st.w)
        return dict(rgb=rgb, grads=dict(zip(ORDER, torch.autograd.grad(rgb, st.leaves, st.grad_rgb))))
    if path == "step":
        st.step.replay()
        return dict(rgb=st.step.st.rgb, loss=st.step.loss, grads={k: st.step.out[k] for k in ORDER})
    if path == "train":
        st.step.replay()
        return dict(rgb=st.step.st.rgb, loss=st.step.loss, grads={k: st.step.flat.grad[k] for k in ORDER})
    if path == "chain":
        st.r.wsr_project(st.g, st.kind, st.w, st.records)
        st.r.wsr_project_bwd(st.g, st.kind, st.w, st.grad_records, st.grads)
        rec = st.records.view(st.r.n_cams, case["n"], A.WSR_RECORD_FLOATS)
        return dict(mean=rec[..., 0:2], conic=rec[..., 2:5], colour=rec[..., 5:9], extent=rec[..., 9:11],
                    depth=rec[..., 11], grads={k: st.out[k] for k in ORDER[:6]})
    if path == "loss":
        st.r.wsr_loss_3dgs(st.rgb, st.target, 0.2, st.loss, st.grad)
        return dict(loss=st.loss, grad=st.grad)
    st.opt.wsr_adam_step()
    return dict(param=st.flat.data, exp_avg=st.opt.exp_avg, exp_avg_sq=st.opt.exp_avg_sq)


# --------------------------------------------------------------------------------------------
# What a pass cannot do without
# --------------------------------------------------------------------------------------------

def _pairs(case):
    """(pixel, Gaussian) pairs inside the footprints, estimated from a sample of the scene's distribution: the
    area of each sampled ellipse, times the part of its box inside the image."""
    rng, m = np.random.default_rng(0), 4000
    if case["spread"] == "box":
        p, mu, sd = rng.uniform(-1, 1, (m, 3)), -3.0, 0.5
    else:
        p, mu, sd = rng.uniform(-3, 3, (m, 3)) + rng.normal(0, 0.3, (m, 3)), -4.0, 0.7
    s2 = np.exp(2 * rng.normal(mu, sd, (m, 3)))
    Q = np.linalg.qr(rng.normal(size=(m, 3, 3)))[0]
    S3 = np.einsum("mij,mj,mkj->mik", Q, s2, Q)
    total = 0.0
    for c in _cameras(case):
        t = p @ c.R.T + c.T
        ok = t[:, 2] > c.znear
        z = np.where(ok, t[:, 2], 1.0)
        lx, ly = 0.65 * c.width / c.fx, 0.65 * c.height / c.fy
        J = np.zeros((m, 2, 3))
        J[:, 0, 0], J[:, 1, 1] = c.fx / z, c.fy / z
        J[:, 0, 2] = -c.fx * np.clip(t[:, 0] / z, -lx, lx) / z
        J[:, 1, 2] = -c.fy * np.clip(t[:, 1] / z, -ly, ly) / z
        T = J @ c.R
        S = T @ S3 @ T.transpose(0, 2, 1) + 0.3 * np.eye(2)
        mean = np.stack([c.fx * t[:, 0] / z + c.cx, c.fy * t[:, 1] / z + c.cy], 1)
        h = 3 * np.sqrt(np.stack([S[:, 0, 0], S[:, 1, 1]], 1))
        size = np.array([c.width, c.height])
        inside = np.clip(np.minimum(mean + h, size) - np.maximum(mean - h, 0), 0, None) / (2 * h)
        area = 9 * math.pi * np.sqrt(np.maximum(np.linalg.det(S), 0))
        total += float((area * inside.prod(1) * ok).mean())
    return total * case["n"]


def work(case):
    path, n, K = case["path"], case["n"], (case["degree"] + 1) ** 2
    width = 3 + 3 + 4 + 3 * K + (K if case["vd"] else 1) + 1
    if path == "adam":                      # p, g, m, v read; p, m, v written
        return dict(bytes=28.0 * n * width, flops=12.0 * n * width)
    pix = _pixels(case)
    if path == "loss":                      # two images read, one written; the separable 11-tap filters
        return dict(bytes=36.0 * pix, flops=3.0 * 2 * 11 * 2 * (5 + 3) * pix)
    params = n * (12 + (14 if case["reduced"] else 28) + (2 if case["reduced"] else 4) * (width - 11) + 4)
    views = len(_cameras(case))
    if path == "chain":                     # parameters and gradient records read; records and gradients written
        return dict(bytes=params + 4.0 * n * width + n * views * (36.0 + 48.0), flops=1500.0 * n * views)
    pairs = _pairs(case)
    if path == "frame":                     # parameters read; colours and denominators written
        return dict(bytes=params + 16.0 * pix, flops=17.0 * pairs + 500.0 * n * views)
    # parameters read, gradients written; the image's gradient or target read, colours written
    b = dict(bytes=params + 4.0 * n * width + 24.0 * pix, flops=52.0 * pairs + 1500.0 * n * views)
    if path == "train":                     # and the optimiser's state and update
        b["bytes"] += 24.0 * n * width
        b["flops"] += 12.0 * n * width + 528.0 * pix
    return b


# --------------------------------------------------------------------------------------------
# The same in float64
# --------------------------------------------------------------------------------------------

def _sh_basis(d, degree):
    x, y, z = d.unbind(1)
    Y = [torch.full_like(x, math.sqrt(1 / (4 * math.pi)))]
    if degree >= 1:
        c = math.sqrt(3 / (4 * math.pi))
        Y += [-c * y, c * z, -c * x]
    if degree >= 2:
        c = math.sqrt(15 / math.pi) / 2
        Y += [c * x * y, -c * y * z, math.sqrt(5 / math.pi) / 4 * (3 * z * z - 1), -c * x * z,
              c / 2 * (x * x - y * y)]
    if degree >= 3:
        a, b, c = (math.sqrt(k / math.pi) for k in (35 / 32, 105 / 4, 21 / 32))
        Y += [-a * y * (3 * x * x - y * y), b * x * y * z, -c * y * (5 * z * z - 1),
              math.sqrt(7 / math.pi) / 4 * z * (5 * z * z - 3), -c * x * (5 * z * z - 1),
              b / 2 * z * (x * x - y * y), -a * x * (x * x - 3 * y * y)]
    return torch.stack(Y, 1)


def _project64(case, s, c):
    """Mean, covariance entries (a, b, c of [[a, b], [b, c]]), opacity times weight, that times the colour,
    and depth of every Gaussian in one view; what is not ``seen`` contributes nothing."""
    R = torch.tensor(c.R, device="cuda")
    t = s["means"] @ R.T + torch.tensor(c.T, device="cuda")
    depth = t[:, 2]
    front = depth > c.znear
    z = torch.where(front, depth, 1.0)
    lx, ly = 0.65 * c.width / c.fx, 0.65 * c.height / c.fy
    ux, uy = (t[:, 0] / z).clamp(-lx, lx), (t[:, 1] / z).clamp(-ly, ly)
    w, x, y, v = torch.nn.functional.normalize(s["quats"], dim=1).unbind(1)
    rot = torch.stack([1 - 2 * (y * y + v * v), 2 * (x * y - w * v), 2 * (x * v + w * y),
                       2 * (x * y + w * v), 1 - 2 * (x * x + v * v), 2 * (y * v - w * x),
                       2 * (x * v - w * y), 2 * (y * v + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    M = R @ (rot * s["log_scales"].exp()[:, None, :])
    r0 = (c.fx / z)[:, None] * (M[:, 0] - ux[:, None] * M[:, 2])
    r1 = (c.fy / z)[:, None] * (M[:, 1] - uy[:, None] * M[:, 2])
    sigma, beta = s["weight_params"][0], s["weight_params"][1]
    if case["weight"] == "exp":
        factor = torch.exp(-sigma * z ** beta)
    elif case["weight"] == "lc":
        factor = (1 - z / sigma).clamp(min=0.0)
    else:
        factor = torch.ones_like(z)
    seen = front & (factor != 0)
    weight = factor * s["lc_v"] if case["weight"] == "lc" else factor
    Y = _sh_basis(torch.nn.functional.normalize(s["means"] - torch.tensor(-c.R.T @ c.T, device="cuda"), dim=1),
                  case["degree"])
    col = (torch.einsum("nk,nkc->nc", Y, s["sh"]) + 0.5).clamp(min=0.0)
    u = (Y * s["opacity"]).sum(1) if case["vd"] else torch.sigmoid(s["opacity"])
    uw = u * weight
    return dict(mx=c.fx * t[:, 0] / z + c.cx, my=c.fy * t[:, 1] / z + c.cy, a=(r0 * r0).sum(1) + 0.3,
                b=(r0 * r1).sum(1), c=(r1 * r1).sum(1) + 0.3, det=torch.linalg.cross(r0, r1).square().sum(1)
                + 0.3 * ((r0 * r0).sum(1) + (r1 * r1).sum(1)) + 0.09, uw=uw, cuw=col * uw[:, None], depth=depth,
                seen=seen)


def _chunks(p, c, most=12_000_000):
    """The pixels of every footprint's box, about ``most`` at a time: (Gaussians, pixels of each, the place of
    each pair's Gaussian among them, pair x, pair y)."""
    hx, hy = 3 * p["a"].sqrt(), 3 * p["c"].sqrt()
    x0 = (p["mx"] - hx - 0.5).ceil().clamp(0, c.width)
    x1 = (p["mx"] + hx - 0.5).floor().clamp(-1, c.width - 1)
    y0 = (p["my"] - hy - 0.5).ceil().clamp(0, c.height)
    y1 = (p["my"] + hy - 0.5).floor().clamp(-1, c.height - 1)
    w, h = (x1 - x0 + 1).clamp(min=0), (y1 - y0 + 1).clamp(min=0)
    area = torch.where(p["seen"], w * h, 0.0).long()
    ids = area.nonzero()[:, 0]
    ends = area[ids].cumsum(0).cpu()
    lo = 0
    while lo < len(ids):
        base = int(ends[lo - 1]) if lo else 0
        hi = max(lo + 1, int(torch.searchsorted(ends, base + most, right=True)))
        g = ids[lo:hi]
        own = torch.repeat_interleave(torch.arange(len(g), device="cuda"), area[g])
        k = torch.arange(len(own), device="cuda") - (area[g].cumsum(0) - area[g])[own]
        wide = w[g].long()[own]
        yield g, area[g], own, x0[g][own] + (k % wide), y0[g][own] + torch.div(k, wide, rounding_mode="floor")
        lo = hi


def _terms(p, g, own, px, py):
    """e = exp(-q / 2) inside q <= 9, and v = inverse covariance times the pixel's offset."""
    dx, dy = px + 0.5 - p["mx"][g][own], py + 0.5 - p["my"][g][own]
    det = p["det"][g]
    A_, B, C = (p["c"][g] / det)[own], (-p["b"][g] / det)[own], (p["a"][g] / det)[own]
    vx, vy = A_ * dx + B * dy, B * dx + C * dy
    ia = (1 / p["a"][g])[own]
    r = dy - (p["b"][g] / p["a"][g])[own] * dx
    q = C * r * r + ia * dx * dx
    return torch.where(q <= 9.0, torch.exp(-0.5 * q), 0.0), vx, vy


def _forward64(p, c, wp):
    P = c.width * c.height
    num = torch.zeros(P, 3, dtype=torch.float64, device="cuda")
    den = torch.zeros(P, dtype=torch.float64, device="cuda")
    for g, _, own, px, py in _chunks(p, c):
        e, _, _ = _terms(p, g, own, px, py)
        at = (py * c.width + px).long()
        den.index_add_(0, at, p["uw"][g][own] * e)
        for k in range(3):
            num[:, k].index_add_(0, at, p["cuw"][g, k][own] * e)
    den = den + wp[2]
    return (num + wp[3:6] * wp[2]) / den[:, None], den


def _backward64(p, c, rgb, den, G):
    """Gradients for every projected quantity of one view."""
    Gd = G / den[:, None]
    GC = (Gd * rgb).sum(1)
    n = len(p["mx"])
    out = {k: torch.zeros(n, dtype=torch.float64, device="cuda") for k in ("mx", "my", "a", "b", "c", "uw")}
    out["cuw"] = torch.zeros(n, 3, dtype=torch.float64, device="cuda")
    for g, count, own, px, py in _chunks(p, c):
        e, vx, vy = _terms(p, g, own, px, py)
        at = (py * c.width + px).long()
        last = count.cumsum(0) - 1

        def total(x):
            s = x.cumsum(0)[last]
            return torch.diff(s, prepend=s.new_zeros(1))

        for k in range(3):
            out["cuw"][g, k] = total(Gd[:, k][at] * e)
        out["uw"][g] = total(-GC[at] * e)
        de = e * ((Gd[at] * p["cuw"][g][own]).sum(1) - p["uw"][g][own] * GC[at])    # e dL/de
        out["mx"][g] = total(de * vx)
        out["my"][g] = total(de * vy)
        out["a"][g] = total(0.5 * de * vx * vx)
        out["b"][g] = total(de * vx * vy)
        out["c"][g] = total(0.5 * de * vy * vy)
    return out


def _chain64(case, s, grads_of):
    """Gradients of the parameters from ``grads_of(view, camera, projected)``, a dict like ``_backward64``'s."""
    leaves = {k: s[k].detach().requires_grad_() for k in ORDER}
    total = {k: torch.zeros_like(s[k]) for k in ORDER}
    for v, c in enumerate(_cameras(case)):
        p = _project64(case, leaves, c)
        up = grads_of(v, c, {k: x.detach() for k, x in p.items()})
        seen = p["seen"]
        outs = [torch.where(seen if p[k].dim() == 1 else seen[:, None], p[k], 0.0) for k in up]
        got = torch.autograd.grad(outs, [leaves[k] for k in ORDER], list(up.values()), allow_unused=True)
        for k, x in zip(ORDER, got):
            if x is not None:
                total[k] += x
    return total


def _render64(case, s, image_grad):
    """Colours, denominators and, for ``image_grad(rgb)``, gradients, views concatenated."""
    views = []
    with torch.no_grad():
        for c in _cameras(case):
            views.append(_forward64(_project64(case, s, c), c, s["weight_params"]))
    rgb, den = torch.cat([x for x, _ in views]), torch.cat([x for _, x in views])
    if image_grad is None:
        return rgb, den, None
    G, at, wp, bg = image_grad(rgb), 0, s["weight_params"], torch.zeros(6, dtype=torch.float64, device="cuda")
    parts = []
    for r, d in views:
        parts.append(G[at:at + len(d)])
        at += len(d)
        bg[2] += (parts[-1] * (wp[3:6] - r) / d[:, None]).sum()
        bg[3:6] += (parts[-1] * wp[2] / d[:, None]).sum(0)
    with torch.enable_grad():
        grads = _chain64(case, s, lambda v, c, p: _backward64(p, c, views[v][0], views[v][1], parts[v]))
    grads["weight_params"] = grads["weight_params"] + bg
    return rgb, den, grads


def _l1(x, y):
    return (x - y).abs().mean(), torch.sign(x - y) / x.numel()


def _loss64(case, x, y, lam=0.2):
    """{L, L1, SSIM} and dL/dx of the 3DGS loss: 11 x 11 Gaussian window of deviation 1.5, zero padding."""
    k = torch.exp(-(torch.arange(11, dtype=torch.float64, device="cuda") - 5) ** 2 / 4.5)
    k = k / k.sum()
    x = x.detach().requires_grad_()
    total, at = 0.0, 0
    with torch.enable_grad():
        for c in _cameras(case):
            a, b = (t[at:at + c.width * c.height].T.reshape(3, 1, c.height, c.width) for t in (x, y))
            at += c.width * c.height

            def blur(t):
                # the eleven taps as shifted sums, one axis at a time
                p = torch.nn.functional.pad(t, (0, 0, 5, 5))
                t = sum(k[i] * p[:, :, i:i + t.shape[2]] for i in range(11))
                p = torch.nn.functional.pad(t, (5, 5))
                return sum(k[i] * p[..., i:i + t.shape[3]] for i in range(11))

            ma, mb = blur(a), blur(b)
            saa, sbb, sab = blur(a * a) - ma * ma, blur(b * b) - mb * mb, blur(a * b) - ma * mb
            total = total + (((2 * ma * mb + 1e-4) * (2 * sab + 9e-4))
                             / ((ma * ma + mb * mb + 1e-4) * (saa + sbb + 9e-4))).sum()
        ssim = total / x.numel()
        l1, sign = _l1(x.detach(), y)
        grad = (1 - lam) * sign + torch.autograd.grad(lam * (1 - ssim), x)[0]
    ssim = ssim.detach()
    return torch.stack([(1 - lam) * l1 + lam * (1 - ssim), l1, ssim]), grad


def exact(case, seed):
    path = case["path"]
    if case["views"] and _pairs(case) > 1e10:
        return None                         # minutes in float64
    if path == "adam":
        flat, opt = _adam(case)
        _adam_values(case, flat, opt, seed)
        g = flat.grad_data.double()
        m = 0.9 * opt.exp_avg.double() + 0.1 * g
        v = 0.999 * opt.exp_avg_sq.double() + 0.001 * g * g
        rate = torch.zeros_like(m)
        K = (case["degree"] + 1) ** 2
        for k in ORDER:
            lr = {"means": 1.6e-4, "log_scales": 5e-3, "sh": 2.5e-3, "opacity": 5e-2}.get(k, 1e-3)
            r = rate[flat.offsets[k]:flat.offsets[k] + flat.count(k)]
            r.fill_(lr)
            if k == "sh":
                r.view(-1, K, 3)[:, 1:] = lr / 20
            elif k == "opacity" and case["vd"]:
                r.view(-1, K)[:, 1:] = lr / 20
        t = 701
        p = flat.data.double() - rate * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-15)
        at = torch.zeros(flat.numel, dtype=torch.bool, device="cuda")
        for k in ORDER:
            at[flat.offsets[k]:flat.offsets[k] + flat.count(k)] = True      # padding between tensors stays
        return dict(param=p, exp_avg=torch.where(at, m, opt.exp_avg.double()),
                    exp_avg_sq=torch.where(at, v, opt.exp_avg_sq.double()))
    if path == "loss":
        loss, grad = _loss64(case, _image(case, seed, "fit").double(), _image(case, seed, "photo").double())
        return dict(loss=loss, grad=grad)
    s32 = _scene(case, seed)
    s = {k: t.double() for k, t in s32.items()}
    if path == "chain":
        rec, half = [], math.log2(math.e) / 2
        gr = _record_grads(case, s32, seed).view(-1, case["n"], 12).double()

        def frame(p):
            qs = (half * p["a"] / p["det"]).sqrt()
            return qs, -(p["b"] / p["a"]) * qs, half / p["a"]

        def up(v, c, p):
            qs, qw, qd = frame(p)
            Sr, Sx, Srr, Srx, Sxx, guw = gr[v, :, :6].unbind(1)
            return dict(mx=-2 * (qw * Sr + qd * Sx), my=-2 * qs * Sr,
                        a=-(Srr * qw * qw + 2 * qd * Srx * qw + qd * qd * Sxx) / half,
                        b=-2 * (Srr * qw * qs + qd * Srx * qs) / half, c=-Srr * qs * qs / half, uw=guw,
                        cuw=gr[v, :, 6:9])

        for c in _cameras(case):
            p = _project64(case, s, c)
            qs, qw, qd = frame(p)
            r = torch.stack([p["mx"], p["my"], qs, qw, qd, p["uw"], *p["cuw"].T,
                             3 * p["a"].sqrt() * 1.0001 + 0.01, 3 * p["c"].sqrt() * 1.0001 + 0.01, p["depth"]], 1)
            gone = torch.zeros_like(r)
            gone[:, 9:11], gone[:, 11] = -1.0, p["depth"]
            rec.append(torch.where(p["seen"][:, None], r, gone))
        rec = torch.stack(rec)
        with torch.enable_grad():
            grads = _chain64(case, s, up)
        return dict(mean=rec[..., 0:2], conic=rec[..., 2:5], colour=rec[..., 5:9], extent=rec[..., 9:11],
                    depth=rec[..., 11], grads={k: grads[k] for k in ORDER[:6]})
    if path == "frame":
        rgb, den, _ = _render64(case, s, None)
        return dict(rgb=rgb, den=den)
    loss = None
    if path == "grad":
        def image_grad(rgb):
            return _image(case, seed, "grad").double()
    else:
        target = _image(case, seed, "target").double()

        def image_grad(rgb):
            nonlocal loss
            loss, G = _loss64(case, rgb, target) if path == "train" else _l1(rgb, target)
            return G
    rgb, den, grads = _render64(case, s, image_grad)
    if path == "grad":
        return dict(rgb=rgb, grads=grads)
    return dict(rgb=rgb, loss=loss.reshape(-1), grads=grads)
