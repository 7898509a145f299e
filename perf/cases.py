"""The work that users of this framework have it do, as cases to time and to compare.

A case is one call, or one short sequence of calls, that a program makes again and again:
training steps of the rasterizer (forward, L1 loss, gradient) from a thumbnail to four
large views, an iteration of the training loop, a rendered view, a differentiable
render inside someone else's autograd graph, the photometric loss, the optimiser, a
densification event and the energy schedule of a training image.

Scenes come from the generator of `synth.surface_scene` (Gaussians on surface patches
plus a sparse background), drawn on the GPU; cameras are `synth.orbit_camera`s.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2507_20239_gb300 import autograd as A
from paper_2507_20239_gb300 import optim as O
from paper_2507_20239_gb300 import rasterizer as R
from paper_2507_20239_gb300 import schedule as S
from paper_2507_20239_gb300 import step as ST
from paper_2507_20239_gb300 import synth
from paper_2507_20239_gb300 import train as TR

DEV = "cuda"
MIXED = ((0.25, "quarter"), (0.5, "half"), (1.0, "full"))


def _step(name, n, width, height, views=1, degree=3, coeffs=16, backward="splat", mixed=False, scene=1.0):
    return dict(name=name, kind="step", n=n, width=width, height=height, views=views, degree=degree, coeffs=coeffs,
                backward=backward, mixed=mixed, scene=scene)


def listed():
    return [
        # a thumbnail: a couple of thousand Gaussians, one 64 x 64 view, as in quick checks and
        # tests; launches and latency are all there is
        _step("step-2k-64x64", 2_000, 64, 64, degree=0, coeffs=1, backward="pixel"),
        # the coarse start of training: few Gaussians, a quarter-resolution view, low SH
        # degree with all 16 coefficients stored
        _step("step-100k-312x207", 100_000, 312, 207, degree=1, backward="pixel"),
        # the ordinary step at full size: 1.5M Gaussians, SH 3, one 1246 x 826 view
        _step("step-1500k-1246x826", 1_500_000, 1246, 826),
        # a batch of mixed-resolution views (a quarter, a half, full) in one launch per stage
        _step("step-500k-12views", 500_000, 1246, 826, views=12, mixed=True),
        # the largest: 5M Gaussians, four views of 1600 x 1060
        _step("step-5M-4x1600x1060", 5_000_000, 1600, 1060, views=4, scene=3.0),
        # one iteration of the training loop at half resolution: eager autograd, Eq. 3 loss
        # with D-SSIM, sparse Adam
        dict(name="train-300k-623x413", kind="train", n=300_000, width=623, height=413, degree=2, backward="pixel"),
        # a viewer's frame at an odd size: projection, binning and compositing, no gradient
        dict(name="render-600k-979x653", kind="render", n=600_000, width=979, height=653, degree=3, coeffs=16),
        # a differentiable render under another program's loss, ragged sizes, a background
        # colour, SH 2 with exactly its nine coefficients
        dict(name="grad-37777-417x305", kind="grad", n=37_777, width=417, height=305, degree=2, coeffs=9,
             backward="splat"),
        # the photometric loss and its gradient on a full-resolution view
        dict(name="loss-1246x826", kind="loss", width=1246, height=826, views=1),
        # the sparse optimiser step over 1.2M Gaussians
        dict(name="adam-1200k", kind="adam", n=1_200_000, coeffs=16, seen=0.64),
        # a densification event: adaptive pruning, split and clone, moments and provenance carried
        dict(name="densify-1200k", kind="densify", n=1_200_000, coeffs=16, adaptive=True),
        # the energy schedule of one training image, scales 1 to 4
        dict(name="energy-1246x826", kind="energy", width=1246, height=826, scales=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo, hi):
    w = _log(rng, lo, hi)
    return w, max(17, int(w * rng.uniform(0.55, 1.0)))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "train", "render", "grad", "loss", "adam", "densify", "energy"])
    degree = rng.randint(0, 3)
    coeffs = rng.choice([(degree + 1) ** 2, 16])
    if kind == "step":
        n, views = _log(rng, 1_500, 4_000_000), rng.choice([1, 1, 1, 2, 3, 4, 7])
        views = max(1, min(views, 12_000_000 // n))
        w, h = _size(rng, 50, 1600)
        while views * w * h > 6_000_000 or n > 60 * w * h:
            w, h = _size(rng, 50, 1600)
            n = min(n, 50 * w * h)
        return dict(kind=kind, n=n, width=w, height=h, views=views, degree=degree, coeffs=coeffs,
                    backward=rng.choice(["pixel", "splat"]), mixed=views >= 3 and rng.random() < 0.5,
                    scene=3.0 if n > 2_000_000 else 1.0)
    if kind == "train":
        w, h = _size(rng, 150, 1300)
        return dict(kind=kind, n=_log(rng, 20_000, 1_000_000), width=w, height=h, degree=degree,
                    backward=rng.choice(["pixel", "splat"]))
    if kind == "render":
        w, h = _size(rng, 60, 1950)
        return dict(kind=kind, n=_log(rng, 2_000, 3_000_000), width=w, height=h, degree=degree, coeffs=coeffs)
    if kind == "grad":
        w, h = _size(rng, 60, 900)
        return dict(kind=kind, n=_log(rng, 2_000, 300_000), width=w, height=h, degree=degree, coeffs=coeffs,
                    backward=rng.choice(["pixel", "splat"]))
    if kind == "loss":
        w, h = _size(rng, 40, 1950)
        return dict(kind=kind, width=w, height=h, views=rng.choice([1, 1, 2, 4]))
    if kind == "adam":
        return dict(kind=kind, n=_log(rng, 2_000, 5_000_000), coeffs=coeffs, seen=rng.choice([0.3, 0.64, 1.0]))
    if kind == "densify":
        return dict(kind=kind, n=_log(rng, 2_000, 2_500_000), coeffs=coeffs, adaptive=rng.random() < 0.5)
    w, h = _size(rng, 60, 1300)
    return dict(kind=kind, width=w, height=h, scales=rng.randint(1, 6))


# ------------------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _scene(case, seed, coeffs):
    """`synth.surface_scene`'s distributions on the GPU: 90% of the means on 20 square or
    hemispherical patches, 10% in a ball; log-scales N(-4, 0.7), logits N(0, 1)."""
    n, k = case["n"], case.get("scene", 1.0)
    g, rng = _gen(seed), np.random.default_rng(seed)
    norm = lambda *s: torch.randn(*s, generator=g, device=DEV)      # noqa: E731
    unif = lambda *s: torch.rand(*s, generator=g, device=DEV)       # noqa: E731
    quats = torch.nn.functional.normalize(norm(n, 4), dim=1)
    logits = norm(n)
    sh = torch.zeros(n, coeffs, 3, device=DEV)
    sh[:, 0] = unif(n, 3)
    if coeffs > 1:
        sh[:, 1:] = 0.05 * norm(n, coeffs - 1, 3)
    if case["kind"] == "step" and case["width"] <= 128:   # the small scene: a cube of larger Gaussians
        return dict(means=2 * unif(n, 3) - 1, log_scales=-3 + 0.5 * norm(n, 3), quats=quats, opacity_logits=logits,
                    sh=sh)
    planar = rng.uniform(size=20) < 0.5
    half = np.where(planar, rng.uniform(0.3, 1.0, 20), rng.uniform(0.2, 0.8, 20)) * k
    area = np.where(planar, 4.0, 2 * math.pi) * half * half
    centre = rng.standard_normal((20, 3))
    centre *= (2.0 * k * rng.uniform(size=(20, 1)) ** (1 / 3)) / np.linalg.norm(centre, axis=1, keepdims=True)
    axis = rng.standard_normal((20, 3))
    axis /= np.linalg.norm(axis, axis=1, keepdims=True)
    u = np.cross(axis, np.where(np.abs(axis[:, :1]) < 0.9, [[1.0, 0, 0]], [[0, 1.0, 0]]))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    f32 = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32, device=DEV)   # noqa: E731
    p = torch.searchsorted(f32(np.cumsum(area / area.sum())), unif(n)).clamp_(max=19)
    r1, r2 = unif(n, 1), unif(n, 1)
    hp, on = f32(half)[p][:, None], torch.as_tensor(planar, device=DEV)[p][:, None]
    up, ap = f32(u)[p], f32(axis)[p]
    vp = torch.linalg.cross(ap, up)
    cz, phi = r1, 2 * math.pi * r2
    sz = (1 - cz * cz).clamp_(min=0).sqrt()
    off = torch.where(on, hp * ((2 * r1 - 1) * up + (2 * r2 - 1) * vp),
                      hp * (sz * phi.cos() * up + sz * phi.sin() * vp + cz * ap))
    ball = torch.nn.functional.normalize(norm(n, 3), dim=1) * (10.0 * k * unif(n, 1) ** (1 / 3))
    means = torch.where(unif(n, 1) < 0.1, ball, f32(centre)[p] + off)
    return dict(means=means.contiguous(), log_scales=-4 + 0.7 * norm(n, 3), quats=quats, opacity_logits=logits, sh=sh)


def _cameras(case, seed):
    views, w, h, k = case.get("views", 1), case["width"], case["height"], case.get("scene", 1.0)
    az = np.random.default_rng(seed + 7).uniform(0, 2 * math.pi)
    if case["kind"] == "step" and w <= 128:
        return [synth.orbit_camera(4.0, az + 2 * math.pi * v / views, 0.0, w, h, float(w)) for v in range(views)]
    out = []
    for v in range(views):
        s = MIXED[v % 3][0] if case.get("mixed") else 1.0
        out.append(synth.orbit_camera(4.0 * k, az + 2 * math.pi * v / views, 15.0, max(8, round(w * s)),
                                      max(8, round(h * s)), w * s))
    return out


def _targets(cams, seed):
    g = _gen(seed + 1)
    return [torch.rand(3, c.height, c.width, generator=g, device=DEV) for c in cams]


def _picture(views, h, w, seed):
    """Images with large-scale structure and fine noise, and targets near them."""
    g = _gen(seed)
    low = torch.rand(views, 3, 12, 16, generator=g, device=DEV)
    big = torch.nn.functional.interpolate(low, size=(h, w), mode="bicubic", align_corners=False)
    noisy = lambda a: (big + a * torch.randn(views, 3, h, w, generator=g, device=DEV)).clamp_(0, 1)   # noqa: E731
    return noisy(0.04), noisy(0.02)


def _moments(params, seed):
    """Adam moments of a training run under way: |gradients| of 1e-7 to 1e-5."""
    g = _gen(seed + 3)
    out = {}
    for k in R.PARAM_KEYS:
        s = 10.0 ** (2 * torch.rand(params[k].shape, generator=g, device=DEV) - 7)
        out[k + ".v"] = (s * s).reshape(len(s), -1)
        out[k + ".m"] = (s * torch.randn(params[k].shape, generator=g, device=DEV)).reshape(len(s), -1)
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "step":
        P, cams = _scene(case, seed, case["coeffs"]), _cameras(case, seed)
        st = ST.TrainStep(P, case["degree"], cams, _targets(cams, seed), ST.StepConfig(backward=case["backward"]))
        graph = st.capture()
        st.stats.accum.zero_()
        st.stats.count.zero_()
        return dict(kind=kind, step=st, graph=graph)
    if kind == "train":
        P, cams = _scene(case, seed, 16), _cameras(case, seed)
        sched = TR.Schedule(stages=[(0, 2, R.DENSIFY_SPLIT_ONLY), (20_000, 1, R.DENSIFY_ADAPTIVE)], total=30_000,
                            sh_every=1000, backward=case["backward"])
        tr = TR.Trainer({k: v.cpu().numpy() for k, v in P.items()},
                        {2: (cams, [t.cpu().numpy() for t in _targets(cams, seed)])}, sched, extent=4.4)
        tr.opt.set_moments(_moments(P, seed), P)
        tr.opt.t = 2000
        return dict(kind=kind, trainer=tr, it=1000 * case["degree"] + 500)
    if kind in ("render", "grad"):
        P, cams = _scene(case, seed, case["coeffs"]), _cameras(case, seed)
        state = dict(kind=kind, P=P, frame=R.Frame(cams), degree=case["degree"])
        if kind == "grad":
            w, h = case["width"], case["height"]
            state.update(backward=case["backward"],
                         d_image=torch.randn(3 * w * h, generator=_gen(seed + 2), device=DEV) / (3 * w * h))
            for k in R.PARAM_KEYS:
                P[k].requires_grad_(True)
        return state
    if kind == "loss":
        w, h, views = case["width"], case["height"], case["views"]
        image, target = _picture(views, h, w, seed)
        cams = [synth.orbit_camera(4.0, 0.1 + v, 15.0, w, h, float(w)) for v in range(views)]
        return dict(kind=kind, frame=R.Frame(cams), image=image.reshape(-1), target=target.reshape(-1))
    if kind == "adam":
        n = case["n"]
        P = _scene(case, seed, case["coeffs"])
        mom, g = _moments(P, seed), _gen(seed + 5)
        grads = {k: (mom[k + ".v"].sqrt() * torch.randn(mom[k + ".v"].shape, generator=g, device=DEV)).reshape(P[k].shape)
                 for k in R.PARAM_KEYS}
        opt = O.Adam(P, TR.default_lrs(4.4))
        opt.set_moments(mom, P)
        opt.t = 2000
        radius = None
        if case["seen"] < 1.0:
            radius = torch.where(torch.rand(n, generator=g, device=DEV) < case["seen"],
                                 torch.randint(1, 60, (n,), generator=g, device=DEV), 0).to(torch.int32)
        return dict(kind=kind, P=P, opt=opt, grads=grads, radius=radius)
    if kind == "densify":
        n = case["n"]
        P, g = _scene(case, seed, case["coeffs"]), _gen(seed + 6)
        count = torch.randint(0, 100, (n,), generator=g, device=DEV, dtype=torch.int32)
        accum = count * 10.0 ** (2.2 * torch.rand(n, generator=g, device=DEV) - 5.7)
        lg = lambda p: math.log(p / (1 - p))    # noqa: E731
        prune = dict(prune_ratio=0.02, prune_upper_logit=lg(0.05)) if case["adaptive"] else dict(prune_logit=lg(0.005))
        cfg = R.densify_cfg(mode=R.DENSIFY_ADAPTIVE, log_scale_threshold=math.log(0.044), seed=3, event=5, **prune)
        prov = dict(origin=torch.arange(n, dtype=torch.int32, device=DEV),
                    splits=torch.randint(0, 4, (n,), generator=g, device=DEV, dtype=torch.int32),
                    clones=torch.randint(0, 4, (n,), generator=g, device=DEV, dtype=torch.int32))
        # the other buffer set, which a program that keeps two swaps with this one: room for 30% growth
        extra, cap = _moments(P, seed), int(1.3 * n) + 64
        room = lambda t: torch.zeros((cap,) + tuple(t.shape[1:]), dtype=t.dtype, device=DEV)    # noqa: E731
        return dict(kind=kind, P=P, cfg=cfg, accum=accum, count=count, extra=extra, prov=prov, cap=cap,
                    out={k: room(t) for k, t in {**P, **prov}.items()}, ex_out={k: room(t) for k, t in extra.items()},
                    degree=int(round(math.sqrt(case["coeffs"]))) - 1)
    image, _ = _picture(1, case["height"], case["width"], seed)
    return dict(kind=kind, image=image[0].cpu().numpy(), scales=case["scales"])


# ---------------------------------------------------------------------------------- run
def run(s):
    kind = s["kind"]
    if kind == "step":
        s["graph"].replay()
        st = s["step"]
        return dict(image=st.image, T=st.T, loss=st.loss, grads=st.pgrads, accum=st.stats.accum, count=st.stats.count,
                    radius=st.proj.radius)
    if kind == "train":
        tr = s["trainer"]
        loss = tr.step(s["it"])
        return dict(loss=loss, params={k: tr.P[k].detach() for k in R.PARAM_KEYS}, m=tr.opt.m, v=tr.opt.v,
                    accum=tr.stats.accum, count=tr.stats.count)
    if kind == "render":
        proj = R.project(s["P"], s["degree"], s["frame"])
        bins = R.bin_sort(proj, s["frame"])
        image, T, _ = R.raster_fwd(proj, bins, s["frame"])
        return dict(image=image, T=T, entries=bins.count)
    if kind == "grad":
        P = s["P"]
        for k in R.PARAM_KEYS:
            P[k].grad = None
        image, T = A.rasterize(P, s["degree"], s["frame"], bg=(0.2, 0.5, 1.0), backward=s["backward"])
        image.backward(s["d_image"])
        return dict(image=image.detach(), T=T, grads={k: P[k].grad for k in R.PARAM_KEYS})
    if kind == "loss":
        d_image, loss = O.photometric_loss_grad(s["frame"], s["image"], s["target"], 0.2)
        return dict(d_image=d_image, loss=loss)
    if kind == "adam":
        s["opt"].step(s["P"], s["grads"], radius=s["radius"])
        return dict(params=s["P"], m=s["opt"].m, v=s["opt"].v)
    if kind == "densify":
        split, clone, tau, new_n, ws = R.densify_select(s["cfg"], s["P"], s["accum"], s["count"])
        out, extra, got, err = R.densify_apply(s["cfg"], s["P"], s["degree"], split, clone, tau, s["cap"],
                                               extra=s["extra"], ws=ws, out=s["out"], ex_out=s["ex_out"],
                                               prov=s["prov"])
        return dict(split=split, clone=clone, tau=tau, new_n=new_n, out=out, extra=extra, got=got, err=err)
    return dict(E=S.energies([s["image"]], s["scales"]))


# --------------------------------------------------------------------------------- work
def _pixels(case):
    w, h, views = case["width"], case["height"], case.get("views", 1)
    if not case.get("mixed"):
        return w * h * views
    return sum(round(w * MIXED[v % 3][0]) * round(h * MIXED[v % 3][0]) for v in range(views))


def work(case):
    """Bytes: each input read once, each output written once. Operations: the compositing's, from
    the pairs of pixel and Gaussian that it examines (16 operations each way) and composites (10
    forward, 46 backward); about 270 and 140 a pixel where the scene is dense."""
    kind = case["kind"]
    if kind == "energy":
        b = f = 0
        for r in range(1, case["scales"] + 1):
            w, h = max(1, int(case["width"] / r + 0.5)), max(1, int(case["height"] / r + 0.5))
            b += 4 * 3 * w * h
            f += 3 * w * h * 2.5 * math.log2(max(2, w * h))
        return dict(bytes=b, flops=f)
    if kind == "loss":
        px = 3 * _pixels(case)
        return dict(bytes=12 * px, flops=px * (2 * 11 * 2 * 8 + 60))
    n, row = case["n"], 4 * (11 + 3 * case.get("coeffs", 16))
    if kind == "adam":
        return dict(bytes=n * row * (1 + 6 * case["seen"]), flops=n * row / 4 * 12 * case["seen"])
    if kind == "densify":
        return dict(bytes=2 * n * (3 * row + 12) + 10 * n, flops=20 * n)
    px = _pixels(case)
    views = case.get("views", 1)
    dense = min(1.0, views * n * 4 / px)
    if kind == "render":
        return dict(bytes=n * row + 16 * px, flops=px * dense * (270 * 16 + 140 * 10))
    b = 2 * n * row + 24 * px + (6 * n * row if kind == "train" else 0)
    return dict(bytes=b, flops=px * dense * (270 * 32 + 140 * 56))


# -------------------------------------------------------------------------------- exact
def _sh_basis(d, degree):
    x, y, z = d.unbind(1)
    pi = math.pi
    c1, c2 = math.sqrt(3 / (4 * pi)), math.sqrt(15 / pi)
    out = [torch.full_like(x, 0.5 / math.sqrt(pi))]
    if degree >= 1:
        out += [-c1 * y, c1 * z, -c1 * x]
    if degree >= 2:
        out += [c2 / 2 * x * y, -c2 / 2 * y * z, math.sqrt(5 / pi) / 4 * (3 * z * z - 1), -c2 / 2 * x * z,
                c2 / 4 * (x * x - y * y)]
    if degree >= 3:
        a, b, c, e = (math.sqrt(35 / (2 * pi)) / 4, math.sqrt(105 / pi), math.sqrt(21 / (2 * pi)) / 4,
                      math.sqrt(7 / pi) / 4)
        out += [-a * y * (3 * x * x - y * y), b / 2 * x * y * z, -c * y * (5 * z * z - 1), e * z * (5 * z * z - 3),
                -c * x * (5 * z * z - 1), b / 4 * z * (x * x - y * y), -a * x * (x * x - 3 * y * y)]
    return torch.stack(out, 1)


def _records(P, degree, cam):
    """Eq. 1 and the EWA projection in 64 bits: (indices in depth order, records [m, 9] = (u, v, A, beta, gamma, o, rgb),
    half-extents)."""
    f64 = lambda a: torch.as_tensor(np.asarray(a, np.float64), device=DEV)   # noqa: E731
    W, t = f64(cam.R), f64(cam.t)
    tc = P["means"] @ W.T + t
    with torch.no_grad():
        o = torch.sigmoid(P["opacity_logits"])
        i = torch.nonzero((tc[:, 2] > np.float64(np.float32(cam.near))) & (o >= 1 / 255)).squeeze(1)
        i = i[torch.argsort(tc[i, 2], stable=True)]
    tc, o = tc[i], torch.sigmoid(P["opacity_logits"][i])
    w, x, y, z = torch.nn.functional.normalize(P["quats"][i], dim=1).unbind(1)
    rot = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y), 2 * (x * y + w * z),
                       1 - 2 * (x * x + z * z), 2 * (y * z - w * x), 2 * (x * z - w * y), 2 * (y * z + w * x),
                       1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    M = rot * P["log_scales"][i].exp()[:, None, :]
    tz = tc[:, 2]
    lx, ly = 1.3 * 0.5 * cam.width / cam.fx, 1.3 * 0.5 * cam.height / cam.fy
    rx, ry, zero = (tc[:, 0] / tz).clamp(-lx, lx), (tc[:, 1] / tz).clamp(-ly, ly), torch.zeros_like(tz)
    J = torch.stack([cam.fx / tz, zero, -cam.fx * rx / tz, zero, cam.fy / tz, -cam.fy * ry / tz], 1).view(-1, 2, 3)
    K = J @ W @ M
    a, b, c = (K[:, 0] ** 2).sum(1) + 0.3, (K[:, 0] * K[:, 1]).sum(1), (K[:, 1] ** 2).sum(1) + 0.3
    d = torch.nn.functional.normalize(P["means"][i] + W.T @ t, dim=1)
    k = (degree + 1) ** 2
    rgb = ((_sh_basis(d, degree)[:, :, None] * P["sh"][i][:, :k]).sum(1) + 0.5).clamp(min=0)
    rec = torch.cat([torch.stack([cam.fx * tc[:, 0] / tz + cam.cx, cam.fy * tc[:, 1] / tz + cam.cy, c / (a * c - b * b),
                                  -b / c, 1 / c, o], 1), rgb], 1)
    q = 2 * torch.log(255 * o.detach()) + 1e-6
    return i, rec, ((q * a.detach()).clamp(min=0).sqrt(), (q * c.detach()).clamp(min=0).sqrt())


def _composite(rec, px, py, bg):
    """Eq. 2 of depth-ordered records at the pixel centres (px, py): (image [3, p], T [p])."""
    u, v, cA, be, ga, o = (rec[:, k][:, None] for k in range(6))
    dy = v - py
    t = u - px + be * dy
    alpha = (o * torch.exp(-0.5 * (cA * t * t + ga * dy * dy))).clamp(max=0.99)
    alpha = torch.where(alpha >= float(np.float32(1) / np.float32(255)), alpha, 0.0)
    logs = torch.log1p(-alpha)
    after = torch.cumsum(logs, 0)
    go = after.detach() >= math.log(1e-4)
    w = torch.where(go, alpha * torch.exp(after - logs), 0.0)
    T = torch.exp(torch.where(go, logs, 0.0).sum(0))
    return rec[:, 6:].T @ w + T * torch.tensor(bg, dtype=torch.float64, device=DEV)[:, None], T


def _exact_view(P, degree, cam, bg=(0.0, 0.0, 0.0), d_image=None, target=None):
    """One view in 64 bits, tile by tile: the image and T; with d_image or an L1 target, its gradient's
    flow into the records and from there into P[...].grad. Also the records' mean gradients."""
    W, H = cam.width, cam.height
    i, rec, (hx, hy) = _records(P, degree, cam)
    leaf = rec.detach()
    image, T = torch.empty(3, H, W, dtype=torch.float64, device=DEV), torch.empty(H, W, dtype=torch.float64, device=DEV)
    grad = target is not None or d_image is not None
    d_rec = torch.zeros_like(leaf)
    loss = 0.0
    x0s, x1s, y0s, y1s = leaf[:, 0] - hx, leaf[:, 0] + hx, leaf[:, 1] - hy, leaf[:, 1] + hy
    for y0 in range(0, H, 16):
        band = torch.nonzero((y1s >= y0) & (y0s <= y0 + 16)).squeeze(1)
        for x0 in range(0, W, 16):
            y1, x1 = min(y0 + 16, H), min(x0 + 16, W)
            sel = band[(x1s[band] >= x0) & (x0s[band] <= x0 + 16)]
            py, px = torch.meshgrid(torch.arange(y0, y1, device=DEV, dtype=torch.float64) + 0.5,
                                    torch.arange(x0, x1, device=DEV, dtype=torch.float64) + 0.5, indexing="ij")
            part = leaf[sel].requires_grad_(grad)
            img, t = _composite(part, px.reshape(1, -1), py.reshape(1, -1), bg)
            img = img.view(3, y1 - y0, x1 - x0)
            image[:, y0:y1, x0:x1], T[y0:y1, x0:x1] = img.detach(), t.detach().view(y1 - y0, x1 - x0)
            if grad:
                if d_image is not None:
                    d = d_image[:, y0:y1, x0:x1]
                else:
                    diff = img.detach() - target[:, y0:y1, x0:x1]
                    loss = loss + diff.abs().sum() / (3 * W * H)
                    d = diff.sign() / (3 * W * H)
                if len(sel):
                    d_rec.index_add_(0, sel, torch.autograd.grad(img, part, d)[0])
    if not grad:
        return image, T, None, None
    rec.backward(d_rec)
    mean_grad = torch.zeros(P["means"].shape[0], 2, dtype=torch.float64, device=DEV)
    mean_grad[i] = d_rec[:, :2]
    return image, T, loss, mean_grad


def _tiles(case):
    return _pixels(case) / 256


def _exact_ssim(image, target, lam):
    w = torch.exp(-(torch.arange(11, dtype=torch.float64, device=DEV) - 5) ** 2 / (2 * 1.5 ** 2))
    w = w / w.sum()
    win = lambda a: torch.nn.functional.conv2d(torch.nn.functional.conv2d(      # noqa: E731
        a[:, None], w.view(1, 1, 1, 11), padding=(0, 5)), w.view(1, 1, 11, 1), padding=(5, 0))[:, 0]
    x, y = image.double().requires_grad_(True), target.double()
    mx, my = win(x), win(y)
    sxx, syy, sxy = win(x * x) - mx * mx, win(y * y) - my * my, win(x * y) - mx * my
    c1, c2 = 0.01 ** 2, 0.03 ** 2
    ssim = ((2 * mx * my + c1) * (2 * sxy + c2) / ((mx * mx + my * my + c1) * (sxx + syy + c2))).mean()
    loss = (1 - lam) * (x - y).abs().mean() + lam * (1 - ssim)
    return torch.autograd.grad(loss, x)[0], loss.detach()


def _shrink(n_in, n_out):
    """D_r along one axis as a matrix [n_out, n_in]."""
    s = n_in / n_out
    c = (torch.arange(n_out, dtype=torch.float64, device=DEV)[:, None] + 0.5) * s - 0.5
    m = (1 - (torch.arange(n_in, dtype=torch.float64, device=DEV)[None] - c).abs() / s).clamp(min=0)
    return m / m.sum(1, keepdim=True)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("step", "render", "grad"):
        if _tiles(case) > 5000 or case["n"] * case.get("views", 1) > 2_000_000:
            return None
        P = {k: v.double().requires_grad_(True) for k, v in _scene(case, seed, case["coeffs"]).items()}
        cams = _cameras(case, seed)
        if kind == "render":
            with torch.no_grad():
                image, T, _, _ = _exact_view(P, case["degree"], cams[0])
            return dict(image=image.reshape(-1), T=T.reshape(-1), entries=None)
        if kind == "grad":
            w, h = case["width"], case["height"]
            d = (torch.randn(3 * w * h, generator=_gen(seed + 2), device=DEV) / (3 * w * h)).double().view(3, h, w)
            image, T, _, _ = _exact_view(P, case["degree"], cams[0], bg=(0.2, 0.5, 1.0), d_image=d)
            return dict(image=image.reshape(-1), T=T.reshape(-1), grads={k: P[k].grad for k in R.PARAM_KEYS})
        images, Ts, losses, accum = [], [], [], torch.zeros(case["n"], dtype=torch.float64, device=DEV)
        for cam, target in zip(cams, _targets(cams, seed)):
            image, T, loss, mg = _exact_view(P, case["degree"], cam, target=target.double())
            images.append(image.reshape(-1)), Ts.append(T.reshape(-1)), losses.append(loss)
            accum += (mg * torch.tensor([cam.width / 2, cam.height / 2], dtype=torch.float64, device=DEV)).norm(dim=1)
        return dict(image=torch.cat(images), T=torch.cat(Ts), loss=torch.stack(losses),
                    grads={k: P[k].grad for k in R.PARAM_KEYS}, accum=accum, count=None, radius=None)
    if kind == "loss":
        image, target = _picture(case["views"], case["height"], case["width"], seed)
        both = [_exact_ssim(a, b, 0.2) for a, b in zip(image, target)]
        return dict(d_image=torch.cat([d.reshape(-1) for d, _ in both]), loss=torch.stack([v for _, v in both]))
    if kind == "adam":
        s = prepare(case, seed)
        lrs, t = TR.default_lrs(4.4), 2001
        seen = torch.ones(case["n"], dtype=torch.bool, device=DEV) if s["radius"] is None else s["radius"] > 0
        out = dict(params={}, m={}, v={})
        for k in R.PARAM_KEYS:
            p, m, v, g = (a[k].double() for a in (s["P"], s["opt"].m, s["opt"].v, s["grads"]))
            keep = seen.view(-1, *[1] * (p.dim() - 1))
            m2, v2 = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            p2 = p - lrs[k] / (1 - 0.9 ** t) * m2 / (v2.sqrt() / math.sqrt(1 - 0.999 ** t) + 1e-15)
            out["params"][k], out["m"][k], out["v"][k] = (torch.where(keep, b, a) for a, b in ((p, p2), (m, m2), (v, v2)))
        return out
    if kind == "energy":
        image = torch.as_tensor(prepare(case, seed)["image"], device=DEV).double()
        E = []
        for r in range(1, case["scales"] + 1):
            h, w = (max(1, (2 * v + r) // (2 * r)) for v in image.shape[1:])
            small = _shrink(image.shape[1], h) @ image @ _shrink(image.shape[2], w).T if r > 1 else image
            E.append(float(torch.fft.fft2(small).abs().sum()) * r * r)
        return dict(E=np.array(E))
    return None     # the training loop's iteration, and the densification's copies
