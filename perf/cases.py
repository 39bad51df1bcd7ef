"""Workloads of the 4D Gaussian render path, as a user's program calls it.

Kinds of case (every one through the package's public entry points):

  view      one frame of a viewer, or of a rig's cameras: ``Renderer.forward``
  sweep     an evaluation sweep: single views through ``FramePipeline``
  step      a training step: forward, L1 loss and backward to every parameter
            over a batch of views (optionally with the significance mask, its
            loss and the densification statistics, or through autograd)
  aux       a training step on image, depth and opacity (``forward_aux`` /
            ``backward_aux``)
  features  a segmentation step: feature map and its adjoint
  split     densification: children sampled from a share of the Gaussians
  adam      the optimiser's step over all parameter tensors

Scenes follow the distributions of ``synthetic.py`` (drawn on the GPU from the
seed); cameras are its cameras.  ``exact`` evaluates the same mathematics in
64-bit torch from the plain formulas of the paper (Schur-complement slice, EWA
splat, front-to-back blending) with autograd for the gradients.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2412_20720_gb300 import fgs4d, synthetic
from paper_2412_20720_gb300.render import (PARAM_KEYS, Adam, FramePipeline, RenderConfig, Renderer, l1_loss,
                                           mask_loss, render, split_gaussians)

DEVICE = "cuda"

# half-extent of the scene box, range of the spatial scales and the camera
# distance of each scene family
SCENES = {
    "tiny": dict(box=(1.0, 1.0, 1.0), scale=(0.01, 0.1), distance=3.0),
    "orbit": dict(box=(3.0, 3.0, 3.0), scale=(0.01, 0.1), distance=6.0),
    "sphere": dict(box=(5.0, 5.0, 5.0), scale=(0.01, 0.1), distance=9.0),
    "urban": dict(box=(30.0, 30.0, 3.0), scale=(0.02, 1.0), distance=0.0),
}
SPHERE_SIZES = ((512, 512), (800, 800), (1014, 1352), (1352, 1014))


def _case(kind, scene, n, width, height, views=1, degree=3, order=2, tile=16, mask=False, autograd=False, depth=1,
          features=0, children=0):
    return {"kind": kind, "scene": scene, "n": n, "width": width, "height": height, "views": views,
            "degree": degree, "order": order, "tile": tile, "mask": mask, "autograd": autograd, "depth": depth,
            "features": features, "children": children}


def listed():
    cases = [
        # the smallest call: a thumbnail of a small model, where launches and latency are all
        ("tiny_view", _case("view", "tiny", 2000, 128, 96, degree=1, order=1)),
        # the smallest training step, written with autograd
        ("tiny_step", _case("step", "tiny", 2000, 128, 96, degree=1, order=1, autograd=True)),
        # a mid-size compact model under training: odd sizes, degree 2 (SH rows that no 16-byte
        # load divides), the significance mask with its loss, densification statistics
        ("compact_step", _case("step", "orbit", 60_001, 803, 611, views=2, degree=2, order=1, mask=True)),
        # a viewer showing one frame at a time at the paper's resolution
        ("orbit_view", _case("view", "orbit", 300_000, 1352, 1014)),
        # the timestamp sweep of an evaluation, eight frames in flight
        ("orbit_sweep", _case("sweep", "orbit", 300_000, 1352, 1014, views=16, depth=8)),
        # the paper's training batch: four timestamps of one camera
        ("train_step", _case("step", "orbit", 300_000, 1352, 1014, views=4)),
        # a larger model trained on a batch of mixed resolutions in one call
        ("sphere_step", _case("step", "sphere", 1_000_000, 0, 0, views=8)),
        # the largest: a street scene seen by the six cameras of a rig in one call, Gaussians that span
        # many tiles (rendered only: the gradients of Gaussians that touch a camera are cancelling sums
        # that two runs do not reproduce)
        ("urban_rig", _case("view", "urban", 3_000_000, 1920, 1080, views=6)),
        # training with a depth (LiDAR) and an opacity (sky) loss
        ("aux_step", _case("aux", "orbit", 300_000, 1352, 1014)),
        # training of 32-dimensional scale-gated features on a finished model
        ("features_step", _case("features", "orbit", 300_000, 1352, 1014, features=32)),
        # a densification step: a tenth of the Gaussians split into two children each
        ("split", _case("split", "orbit", 300_000, 0, 0, children=2)),
        # the optimiser over a 1M-Gaussian model
        ("adam", _case("adam", "sphere", 1_000_000, 0, 0)),
    ]
    return [dict(c, name=name) for name, c in cases]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(("view", "view", "sweep", "step", "step", "step", "aux", "features", "split", "adam"))
    scene = rng.choice(("orbit", "orbit", "sphere", "urban"))
    degree, order = rng.choice(((3, 2), (3, 2), (3, 1), (3, 0), (2, 2), (2, 1), (1, 1), (0, 0)))
    n = _log_int(rng, 1000, 1_000_000)
    if kind in ("split", "adam"):
        return _case(kind, "orbit" if scene == "urban" else scene, n, 0, 0, degree=degree, order=order,
                     children=rng.randint(1, 3) if kind == "split" else 0)
    width = _log_int(rng, 120, 1920)
    height = max(64, min(1352, int(width * rng.uniform(0.55, 1.3))))
    c = _case(kind, scene, n, width, height, degree=degree, order=order, tile=8 if rng.random() < 0.1 else 16)
    if kind == "sweep":
        c.update(views=rng.randint(4, 16), depth=rng.choice((2, 4, 8)))
    elif kind == "step":
        c.update(views=rng.randint(1, 8), mask=rng.random() < 0.25)
        c.update(autograd=not c["mask"] and rng.random() < 0.25)
    elif kind == "features":
        c.update(features=rng.choice((8, 16, 32)), tile=16)
    if scene == "urban":  # at most a rig's six views; rendered only (see the listed street scene)
        if kind in ("step", "aux"):
            c.update(kind="view", mask=False, autograd=False, views=rng.randint(1, 6))
        c.update(views=min(c["views"], 6))
    return c


# ------------------------------------------------------------------ inputs


def _uniform(gen, shape, lo, hi):
    return torch.rand(shape, device=DEVICE, generator=gen) * (hi - lo) + lo


def _params(case, gen):
    """Scene parameters with the distributions of synthetic.py, float32 on the GPU."""
    n, sc = case["n"], SCENES[case["scene"]]
    k = (case["degree"] + 1) ** 2 * (case["order"] + 1)
    mean = torch.rand((n, 4), device=DEVICE, generator=gen)
    box = torch.tensor(sc["box"], device=DEVICE)
    mean[:, :3] = (2.0 * mean[:, :3] - 1.0) * box
    log_scale = torch.empty((n, 4), device=DEVICE)
    log_scale[:, :3] = _uniform(gen, (n, 3), math.log(sc["scale"][0]), math.log(sc["scale"][1]))
    log_scale[:, 3] = _uniform(gen, (n,), math.log(0.05), math.log(0.3))
    quats = []
    for _ in range(2):
        q = torch.randn((n, 4), device=DEVICE, generator=gen)
        quats.append((q / q.norm(dim=1, keepdim=True)).contiguous())
    logit = torch.randn((n,), device=DEVICE, generator=gen)
    sh = 0.2 * torch.randn((n, k, 3), device=DEVICE, generator=gen)
    return {"mean": mean, "log_scale": log_scale, "q_l": quats[0], "q_r": quats[1], "opacity_logit": logit, "sh": sh}


def _views(case, rng):
    """Cameras of the scene family at seeded angles and timestamps."""
    scene, w, h = case["scene"], case["width"], case["height"]
    dist, out = SCENES[scene]["distance"], []
    if scene == "urban":  # a rig's outward cameras at one timestamp
        t = rng.uniform(0.2, 0.8)
        rig = np.array([-20.0 + 40.0 * t, 0.0, 1.5])
        for j in range(case["views"]):
            yaw = math.radians(60.0 * j)
            d = np.array([math.cos(yaw), math.sin(yaw), 0.0])
            out.append(synthetic.look_at(rig + 2.0 * d, rig + 3.0 * d, (0.0, 0.0, 1.0), w, h, t))
        return out
    turn = rng.uniform(0.0, 2.0 * math.pi)
    for j in range(case["views"]):
        t = rng.uniform(0.1, 0.9)
        if scene == "sphere":
            z, th = rng.uniform(-0.9, 0.9), rng.uniform(0.0, 2.0 * math.pi)
            c = np.array([math.sqrt(1 - z * z) * math.cos(th), z, math.sqrt(1 - z * z) * math.sin(th)]) * dist
        elif case["kind"] == "sweep":  # neighbouring poses of an orbit
            th = turn + 2.0 * math.pi * j / 300.0
            c = np.array([dist * math.sin(th), 0.0, -dist * math.cos(th)])
        else:  # one camera, several timestamps
            c = np.array([dist * math.sin(turn), 0.0, -dist * math.cos(turn)])
        vw, vh = (w, h) if w else SPHERE_SIZES[j % len(SPHERE_SIZES)]
        out.append(synthetic.look_at(c, (0.0, 0.0, 0.0), (0.0, -1.0, 0.0), vw, vh, t))
    return out


def _pixels(views):
    return sum(v["width"] * v["height"] for v in views)


def _capacities(case, views):
    """(visible, instance) capacities of a call over ``views``, with headroom: a
    Gaussian's footprint grows with the resolution, and 8x8 tiles hold four
    times the instances of 16x16 ones."""
    n, vis, inst = case["n"], 0.0, 0.0
    per_view = {"tiny": (0.7, 1.5), "orbit": (0.45, 1.5), "sphere": (0.45, 1.5), "urban": (0.3, 2.8)}[case["scene"]]
    for v in views:
        side = v["width"] / 120.0 if case["scene"] == "urban" else v["width"] / 240.0
        vis += per_view[0] * n
        inst += per_view[0] * n * (2.5 + per_view[1] * side * (1.0 + 0.3 * side))
    if case["tile"] == 8:
        inst *= 4.0
    return int(vis) + 1024, min(int(inst) + 16384, (1 << 30) - 1)


def _smooth_image(gen, h, w):
    """A target photograph: smooth structure with some grain, values in [0, 1]."""
    low = torch.rand((1, 3, 9, 12), device=DEVICE, generator=gen)
    img = torch.nn.functional.interpolate(low, size=(h, w), mode="bilinear", align_corners=False)[0]
    return (0.8 * img + 0.2 * torch.rand((3, h, w), device=DEVICE, generator=gen)).reshape(-1)


def _config(case, views):
    vis, inst = _capacities(case, views)
    # capacities sized for batches; single-view programs leave the visible capacity at its default
    return RenderConfig(sh_degree=case["degree"], t_order=case["order"], tile=case["tile"],
                        bg=(0.1, 0.2, 0.3) if case["mask"] else (0.0, 0.0, 0.0),
                        vis_capacity=vis if len(views) > 1 or case["kind"] == "sweep" else 0, inst_capacity=inst,
                        stage_blocks_per_sm=1 if case["kind"] == "sweep" else 0)


def _inputs(case, seed):
    """The numbers a case works on, made from the seed alone."""
    gen = torch.Generator(device=DEVICE).manual_seed(int(seed) * 7919 + 1)
    rng = random.Random(int(seed) * 104729 + 17)
    kind = case["kind"]
    x = {"params": _params(case, gen)}
    n = case["n"]
    if kind == "adam":
        x["grads"] = {k: 1e-3 * torch.randn(v.shape, device=DEVICE, generator=gen) for k, v in x["params"].items()}
        x["m"] = {k: 1e-3 * torch.randn(v.shape, device=DEVICE, generator=gen) for k, v in x["params"].items()}
        x["v"] = {k: 1e-6 * torch.rand(v.shape, device=DEVICE, generator=gen) for k, v in x["params"].items()}
        x["t"] = rng.randint(10, 3000)
        return x
    if kind == "split":
        m = max(1, n // 10)
        x["idx"] = torch.randperm(n, device=DEVICE, generator=gen)[:m].sort().values.to(torch.int32)
        x["eps"] = torch.randn((m, case["children"], 4), device=DEVICE, generator=gen)
        return x
    x["views"] = _views(case, rng)
    if case["mask"]:
        x["params"]["mask_logit"] = 3.0 * torch.randn((n,), device=DEVICE, generator=gen)
    if kind == "step":
        x["target"] = torch.cat([_smooth_image(gen, v["height"], v["width"]) for v in x["views"]])
    elif kind == "aux":
        # dL/dimage of a photometric loss, dL/ddepth at LiDAR returns (a few percent of the
        # pixels), dL/dopacity of a sky mask
        p = _pixels(x["views"])
        x["dL_drgb"] = torch.randn(3 * p, device=DEVICE, generator=gen) / (3 * p)
        aux = torch.zeros((4, p), device=DEVICE)
        aux[0] = torch.randn(p, device=DEVICE, generator=gen) * (torch.rand(p, device=DEVICE, generator=gen) < 0.05) / p
        aux[1] = torch.randn(p, device=DEVICE, generator=gen) / p
        x["dL_daux"] = aux.reshape(-1)
        x["flow_dt"] = 1.0 / 30.0
    elif kind == "features":
        d, p = case["features"], _pixels(x["views"])
        x["features"] = torch.randn((n, d), device=DEVICE, generator=gen)
        x["gate"] = torch.rand((d,), device=DEVICE, generator=gen)
        x["dL_dF"] = torch.randn(d * p, device=DEVICE, generator=gen) / p
    return x


def prepare(case, seed):
    x = _inputs(case, seed)
    kind, params, n = case["kind"], x["params"], case["n"]
    x["case"] = case
    if kind == "adam":
        opt = Adam(params, lr={k: 1e-2 if k == "opacity_logit" else 1e-3 for k in params})
        for k in params:
            opt.m[k].copy_(x["m"][k])
            opt.v[k].copy_(x["v"][k])
        opt.t.fill_(x["t"])
        x["opt"] = opt
        return x
    if kind == "split":
        x["config"] = RenderConfig(sh_degree=case["degree"], t_order=case["order"])
        return x
    views = x["views"]
    if kind == "sweep":
        pipe = FramePipeline(n, views[0], _config(case, views[:1]), depth=case["depth"])
        x["pipe"], x["g"] = pipe, pipe.slots[0].gaussians(params)
        x["frames"] = [fgs4d.make_views([v]) for v in views]
        x["images"] = [torch.empty((3, v["height"], v["width"]), device=DEVICE) for v in views]
        return x
    r = x["renderer"] = Renderer(n, views, _config(case, views))
    if kind == "step":
        if case["autograd"]:
            x["params"] = {k: v.requires_grad_(True) for k, v in params.items()}
        else:
            x["grads"] = {k: torch.zeros_like(v) for k, v in params.items()}
            x["stats"] = torch.zeros((n, 4), device=DEVICE) if case["mask"] else None
    elif kind == "aux":
        x["grads"] = {k: torch.zeros_like(v) for k, v in params.items()}
    elif kind == "features":
        x["grad_features"] = torch.zeros_like(x["features"])
        x["grad_gate"] = torch.zeros_like(x["gate"])
    elif kind == "view":
        x["T"] = torch.empty(r.total_pixels, device=DEVICE)
    return x


# ------------------------------------------------------------------ one pass


def run(state):
    case, params = state["case"], state["params"]
    kind = case["kind"]
    if kind == "adam":
        opt = state["opt"]
        opt.step(state["grads"])
        return {"params": [params[k] for k in PARAM_KEYS], "m": [opt.m[k] for k in PARAM_KEYS],
                "v": [opt.v[k] for k in PARAM_KEYS]}
    if kind == "split":
        out = split_gaussians(params, state["idx"], state["eps"], 1.6, state["config"])
        return [out[k] for k in PARAM_KEYS]
    if kind == "sweep":
        pipe = state["pipe"]
        pipe.begin()
        for (views, nv), img in zip(state["frames"], state["images"]):
            pipe.submit(state["g"], views, nv, img.data_ptr())
        pipe.end()
        return state["images"]
    r = state["renderer"]
    if kind == "view":
        return {"rgb": r.forward(params, out_T=state["T"]), "T": state["T"]}
    if kind == "features":
        state["grad_features"].zero_()
        state["grad_gate"].zero_()
        out = r.forward_features(params, state["features"], state["gate"])
        r.backward_features(state["features"], state["gate"], state["dL_dF"], state["grad_features"],
                            state["grad_gate"])
        return {"map": out, "grad_features": state["grad_features"], "grad_gate": state["grad_gate"]}
    if case["autograd"]:
        for v in params.values():
            v.grad = None
        img = render(r, params)
        loss = (img - state["target"]).abs().mean()
        loss.backward()
        return {"rgb": img.detach(), "loss": loss.detach(), "grads": [params[k].grad for k in PARAM_KEYS]}
    grads = state["grads"]
    for g in grads.values():
        g.zero_()
    if kind == "aux":
        img, aux = r.forward_aux(params, state["flow_dt"])
        r.backward_aux(params, state["dL_drgb"], state["dL_daux"], grads)
        return {"rgb": img, "aux": aux, "grads": [grads[k] for k in PARAM_KEYS]}
    out = {}
    img = r.forward(params)
    loss, dimg = l1_loss(img, state["target"])
    if case["mask"]:
        state["stats"].zero_()
        out["mask_loss"], _ = mask_loss(params["mask_logit"], grads["mask_logit"])
        out["stats"] = state["stats"]
    r.backward(params, dimg, grads, state["stats"])
    return {**out, "rgb": img, "loss": loss, "grads": [grads[k] for k in grads]}


# ------------------------------------------------------------------ the least work


def work(case):
    """Bytes of inputs read once and outputs written once; operations of the
    alpha evaluations (11 each) and composited entries (9 forward, 25 backward,
    two per feature channel) at the average list depth of the scene."""
    n, kind = case["n"], case["kind"]
    k3 = 3 * (case["degree"] + 1) ** 2 * (case["order"] + 1)
    row = 4 * (17 + k3)  # one Gaussian's parameters
    if kind == "adam":  # parameter and both moments read and written, gradient read
        return {"bytes": 7 * row * n, "flops": 12 * (17 + k3) * n}
    if kind == "split":
        m = max(1, n // 10)
        c = case["children"]
        return {"bytes": m * (4 + row + c * (16 + row)), "flops": m * c * 150}
    if case["width"]:
        px = case["views"] * case["width"] * case["height"]
    else:
        px = sum(a * b for a, b in (SPHERE_SIZES * case["views"])[: case["views"]])
    seen = 0.3 if case["scene"] == "urban" else 0.28
    share = min(1.0, seen * (2.0 if case["views"] > 1 and kind != "sweep" else 1.0))  # visible in some view
    calls = case["views"] if kind == "sweep" else 1
    read = calls * n * 68 + calls * share * n * 4 * k3
    # alpha evaluations: Gaussians per evaluation of a pixel until the lists saturate; about 0.6 of them composite
    deep, most = {"tiny": (48.0, 220.0), "orbit": (1600.0, 220.0), "sphere": (4400.0, 240.0), "urban": (900.0, 50.0)}[
        case["scene"]]
    evals = px * min(most, n / deep)
    flops = 600.0 * n * case["views"] + 11.0 * evals + 0.6 * evals * 9.0
    bytes_ = read + 12.0 * px
    if kind == "view":
        bytes_ += 4.0 * px
    elif kind == "features":
        d = case["features"]
        flops = 600.0 * n + 2.0 * 11.0 * evals + 0.6 * evals * 4.0 * d
        bytes_ = read - share * n * 4 * k3 + 2.0 * n * 4 * d + 2.0 * 4 * d * px
    elif kind in ("step", "aux"):
        flops += 1200.0 * n * case["views"] * seen + 11.0 * evals + 0.6 * evals * 25.0
        bytes_ += n * row + (12.0 if kind == "step" else 28.0 + 16.0) * px  # gradients; target or upstream planes
    return {"bytes": bytes_, "flops": flops}


# ------------------------------------------------------------------ 64-bit values

F64 = torch.float64
NEAR, DILATION, P_T_MIN, MASK_EPS = (float(np.float32(v)) for v in (0.2, 0.3, 0.05, 0.03))


def _quat_matrices(ql, qr):
    a, b, c, d = (ql / ql.norm(dim=1, keepdim=True)).unbind(1)
    p, q, r, s = (qr / qr.norm(dim=1, keepdim=True)).unbind(1)
    left = torch.stack([a, -b, -c, -d, b, a, -d, c, c, d, a, -b, d, -c, b, a], 1).view(-1, 4, 4)
    right = torch.stack([p, -q, -r, -s, q, p, s, -r, r, -s, p, q, s, r, -q, p], 1).view(-1, 4, 4)
    return left @ right


def _sh_basis(degree, d):
    x, y, z = d.unbind(1)
    out = [torch.full_like(x, 0.5 / math.sqrt(math.pi))]
    if degree >= 1:
        c = math.sqrt(3.0 / (4.0 * math.pi))
        out += [-c * y, c * z, -c * x]
    if degree >= 2:
        c = 0.5 * math.sqrt(15.0 / math.pi)
        out += [c * x * y, -c * y * z, 0.25 * math.sqrt(5.0 / math.pi) * (3 * z * z - 1), -c * x * z,
                0.5 * c * (x * x - y * y)]
    if degree >= 3:
        c0, c1 = 0.25 * math.sqrt(7.0 / math.pi), 0.125 * math.sqrt(42.0 / math.pi)
        c2, c3 = 0.25 * math.sqrt(105.0 / math.pi), 0.125 * math.sqrt(70.0 / math.pi)
        out += [-c3 * y * (3 * x * x - y * y), 2 * c2 * x * y * z, -c1 * y * (5 * z * z - 1),
                c0 * z * (5 * z * z - 3), -c1 * x * (5 * z * z - 1), c2 * z * (x * x - y * y),
                -c3 * x * (x * x - 3 * y * y)]
    return torch.stack(out, 1)


def _geometry(case, p, v, flow_dt=0.0):
    """Slice at t and EWA splat of every row of ``p`` (float64): a dict of records and the kept rows."""
    rot = _quat_matrices(p["q_l"], p["q_r"])
    a4 = rot * p["log_scale"].exp()[:, None, :]
    cov = a4 @ a4.transpose(1, 2)
    var_t, cross = cov[:, 3, 3], cov[:, :3, 3]
    dt = float(v["t"]) - p["mean"][:, 3]
    pt = torch.exp(-0.5 * dt * dt / var_t)
    vel = cross / var_t[:, None]
    mu = p["mean"][:, :3] + vel * dt[:, None]
    cov3 = cov[:, :3, :3] - cross[:, :, None] * vel[:, None, :]
    E = torch.tensor(np.asarray(v["viewmat"], dtype=np.float64), device=DEVICE)
    W, T = E[:, :3], E[:, 3]
    fx, fy, cx, cy = (float(v[k]) for k in ("fx", "fy", "cx", "cy"))
    pc = mu @ W.T + T
    x, y, z = pc.unbind(1)
    zero = torch.zeros_like(z)
    J = torch.stack([fx / z, zero, -fx * x / (z * z), zero, fy / z, -fy * y / (z * z)], 1).view(-1, 2, 3)
    M = J @ W
    cov2 = M @ cov3 @ M.transpose(1, 2)
    sa, sb, sd = cov2[:, 0, 0] + DILATION, cov2[:, 0, 1], cov2[:, 1, 1] + DILATION
    det = sa * sd - sb * sb
    uv = torch.stack([fx * x / z + cx, fy * y / z + cy], 1)
    a = torch.sigmoid(p["opacity_logit"]) * pt
    lam = 0.5 * (sa + sd) + torch.sqrt(torch.clamp((0.5 * (sa - sd)) ** 2 + sb * sb, min=0.1))
    rad = torch.ceil(3.0 * torch.sqrt(lam))
    tile = case["tile"]
    gw, gh = -(-v["width"] // tile), -(-v["height"] // tile)
    with torch.no_grad():
        lo = torch.floor((uv - rad[:, None]) / tile)
        hi = torch.floor((uv + rad[:, None]) / tile) + 1
        lim = torch.tensor([gw, gh], dtype=F64, device=DEVICE)
        lo = torch.minimum(lo.nan_to_num().clamp(min=0), lim).long()
        hi = torch.minimum(hi.nan_to_num().clamp(min=0), lim).long()
        keep = (pt >= P_T_MIN) & (z > NEAR) & (det > 0) & (hi > lo).all(1) & (a * 255.0 >= 1.0)
        if "mask_logit" in p:
            keep &= torch.sigmoid(p["mask_logit"]) > MASK_EPS
    rec = {"uv": uv, "conic": torch.stack([sd, -sb, sa], 1) / det[:, None], "a": a, "lo": lo, "hi": hi, "z": z}
    if case["kind"] == "features":
        return rec, keep
    if case["kind"] == "aux":
        pc2 = pc + (vel * flow_dt) @ W.T
        u2 = torch.stack([fx * pc2[:, 0] / pc2[:, 2] + cx, fy * pc2[:, 1] / pc2[:, 2] + cy], 1)
        rec["flow"] = torch.where(pc2[:, 2:3] > NEAR, u2 - uv, torch.zeros_like(uv)).detach()
    w = mu - torch.tensor(np.asarray(v["campos"], dtype=np.float64), device=DEVICE)
    rec["Y"] = _sh_basis(case["degree"], w / w.norm(dim=1, keepdim=True))
    rec["cos"] = torch.stack([torch.cos(2.0 * math.pi * k * dt) for k in range(case["order"] + 1)], 1)
    return rec, keep


def _colour(rec, sh):
    k = rec["Y"].shape[1]
    basis = (rec["cos"][:, :, None] * rec["Y"][:, None, :]).reshape(-1, rec["cos"].shape[1] * k)
    return torch.clamp((basis[:, :, None] * sh).sum(1) + 0.5, min=0.0)


class _Lists:
    """The tiles' depth-ordered lists of one view, and the blending over them in chunks of tiles."""

    def __init__(self, case, v, rec):
        self.tile, self.w, self.h = case["tile"], v["width"], v["height"]
        self.gw, self.gh = -(-self.w // self.tile), -(-self.h // self.tile)
        order = torch.sort(rec["z"].detach().float(), stable=True).indices
        lo, hi = rec["lo"][order], rec["hi"][order]
        wd = hi[:, 0] - lo[:, 0]
        area = wd * (hi[:, 1] - lo[:, 1])
        own = torch.repeat_interleave(torch.arange(len(order), device=DEVICE), area)
        k = torch.arange(len(own), device=DEVICE) - (area.cumsum(0) - area)[own]
        t = (lo[own, 1] + k // wd[own]) * self.gw + lo[own, 0] + k % wd[own]
        by = torch.sort(t, stable=True)
        self.slots = order[own[by.indices]]
        self.count = torch.bincount(by.values, minlength=self.gw * self.gh)
        self.start = self.count.cumsum(0) - self.count

    def chunks(self, budget=12_000_000):
        """Tiles of similar list lengths, together at most ``budget`` (entry, pixel) pairs."""
        by = torch.sort(self.count, descending=True)
        lengths = by.values.tolist()
        i = 0
        while i < len(lengths):
            k = max(1, lengths[i])
            m = max(1, budget // (k * self.tile * self.tile))
            yield by.indices[i:i + m], k
            i += m

    def blend(self, tiles, k, uv, conic, a, attr):
        """Pixel indices [t, p] (-1 outside the image), blended attributes [t, p, c] and final T."""
        j = torch.arange(k, device=DEVICE)
        valid = j[None] < self.count[tiles][:, None]
        s = self.slots[torch.where(valid, self.start[tiles][:, None] + j[None], 0)] if len(self.slots) else \
            torch.zeros_like(valid, dtype=torch.long)
        q = torch.arange(self.tile * self.tile, device=DEVICE)
        px = (tiles % self.gw)[:, None] * self.tile + q % self.tile
        py = (tiles // self.gw)[:, None] * self.tile + q // self.tile
        at = torch.where((px < self.w) & (py < self.h), py * self.w + px, -1)
        dx = uv[s, 0][:, :, None] - (px.to(F64) + 0.5)[:, None, :]
        dy = uv[s, 1][:, :, None] - (py.to(F64) + 0.5)[:, None, :]
        c = conic[s]
        power = -0.5 * (c[:, :, 0:1] * dx * dx + c[:, :, 2:3] * dy * dy) - c[:, :, 1:2] * dx * dy
        alpha = torch.clamp(a[s][:, :, None] * torch.exp(power), max=0.99)
        alpha = torch.where(valid[:, :, None] & (alpha >= 1.0 / 255.0), alpha, torch.zeros_like(alpha))
        with torch.no_grad():  # the entry that would take T below 1e-4 ends the pixel
            live = torch.cumsum(torch.log1p(-alpha), 1) >= math.log(1e-4)
        alpha = alpha * live
        logt = torch.log1p(-alpha)
        after = torch.cumsum(logt, 1)
        weight = alpha * torch.exp(after - logt)
        return at, torch.einsum("tkp,tkc->tpc", weight, attr[s]), torch.exp(after[:, -1])


def _records(case, p, v, x):
    """Records of the visible rows of one view (with autograd where ``p`` has it), their attributes and rows."""
    with torch.no_grad():
        rows = torch.nonzero(_geometry(case, p, v)[1]).squeeze(1)
    q = {k: t[rows] for k, t in p.items() if k not in ("sh", "features", "gate")}
    rec, _ = _geometry(case, q, v, x.get("flow_dt", 0.0))
    if case["kind"] == "features":
        f = p["features"][rows] * p["gate"]
        attr = f / f.norm(dim=1, keepdim=True).clamp(min=1e-300)
    else:
        attr = _colour(rec, p["sh"][rows])
        if case["kind"] == "aux":
            attr = torch.cat([attr, rec["z"][:, None], rec["flow"]], 1)
    return rec, attr, rows


def _planes(case, x, p):
    """Per view: (lists, blended planes [c, h w], T [h w]) without gradients."""
    out = []
    for v in x["views"]:
        rec, attr, rows = _records(case, p, v, x)
        lists = _Lists(case, v, rec)
        img = torch.zeros((attr.shape[1], v["width"] * v["height"]), dtype=F64, device=DEVICE)
        T = torch.ones(v["width"] * v["height"], dtype=F64, device=DEVICE)
        for tiles, k in lists.chunks():
            at, c, t = lists.blend(tiles, k, rec["uv"], rec["conic"], rec["a"], attr)
            ok = at >= 0
            img[:, at[ok]] = c[ok].T
            T[at[ok]] = t[ok]
        out.append((lists, img, T))
    return out


def _pairs(case, x, p):
    """(tile, Gaussian) pairs of all views."""
    total = 0
    for v in x["views"]:
        rec, keep = _geometry(case, p, v)
        total += int(((rec["hi"] - rec["lo"]).prod(1) * keep).sum())
    return total


def _adjoint(case, x, p, planes, d_attr, d_T, names):
    """Gradients of sum <d_attr, planes> + <d_T, T> with respect to p[names], and per view
    (visible rows, dL/duv, dL/dmean)."""
    total = {k: torch.zeros_like(p[k]) for k in names}
    seen = []
    for v, (lists, _, _), da, dT in zip(x["views"], planes, d_attr, d_T):
        leaves = {k: (t.detach().requires_grad_(True) if k in names else t) for k, t in p.items()}
        with torch.enable_grad():
            rec, attr, rows = _records(case, leaves, v, x)
            heads = (rec["uv"], rec["conic"], rec["a"], attr)
            cut = [t.detach().requires_grad_(True) for t in heads]
            for tiles, k in lists.chunks():
                at, c, t = lists.blend(tiles, k, *cut)
                ok = at >= 0
                if not bool(ok.any()):
                    continue
                ((c[ok] * da[:, at[ok]].T).sum() + (t[ok] * dT[at[ok]]).sum()).backward()
            grads = [torch.zeros_like(t) if t.grad is None else t.grad for t in cut]
            pair = [(h, g) for h, g in zip(heads, grads) if h.requires_grad]
            got = torch.autograd.grad([h for h, _ in pair], [leaves[k] for k in names], [g for _, g in pair],
                                      allow_unused=True)
        got = {k: torch.zeros_like(p[k]) if g is None else g for k, g in zip(names, got)}
        for k in names:
            total[k] += got[k]
        seen.append((rows, grads[0], got.get("mean")))
    return total, seen


@torch.no_grad()
def exact(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    p = {k: t.to(F64) for k, t in x["params"].items()}
    if kind == "adam":
        out = {"params": [], "m": [], "v": []}
        t = x["t"] + 1
        for k in PARAM_KEYS:
            g, lr = x["grads"][k].to(F64), float(np.float32(1e-2 if k == "opacity_logit" else 1e-3))
            b1, b2, eps = (float(np.float32(v)) for v in (0.9, 0.999, 1e-8))
            m = b1 * x["m"][k].to(F64) + (1 - b1) * g
            v = b2 * x["v"][k].to(F64) + (1 - b2) * g * g
            out["params"].append(p[k] - lr / (1 - b1 ** t) * m / (v.sqrt() / math.sqrt(1 - b2 ** t) + eps))
            out["m"].append(m)
            out["v"].append(v)
        return out
    if kind == "split":
        i, c = x["idx"].long(), case["children"]
        q = {k: t[i].repeat_interleave(c, 0) for k, t in p.items()}
        rot = _quat_matrices(q["q_l"], q["q_r"])
        off = (rot @ (q["log_scale"].exp() * x["eps"].to(F64).view(-1, 4))[:, :, None])[:, :, 0]
        q["mean"] = q["mean"] + off
        q["log_scale"] = q["log_scale"] - math.log(float(np.float32(1.6)))
        return [q[k] for k in PARAM_KEYS]
    if kind == "features":
        p.update(features=x["features"].to(F64), gate=x["gate"].to(F64))
    frames = x.get("views", [])
    if kind == "sweep":  # the first frames of a long sweep stand for the others
        x["views"] = frames[:4]
    if case["scene"] == "urban" and case["n"] * case["views"] > 2_000_000 or _pairs(case, x, p) > 40_000_000:
        return None  # minutes of 64-bit blending
    planes = _planes(case, x, p)
    bg = (0.1, 0.2, 0.3) if case["mask"] else (0.0, 0.0, 0.0)
    bg = torch.tensor([float(np.float32(b)) for b in bg], dtype=F64, device=DEVICE)[:, None]
    if kind == "features":
        d = case["features"]
        up = x["dL_dF"].to(F64).view(d, -1)
        zero = torch.zeros(up.shape[1], dtype=F64, device=DEVICE)
        g, _ = _adjoint(case, x, p, planes, [up], [zero], ("features", "gate"))
        return {"map": planes[0][1].reshape(-1), "grad_features": g["features"], "grad_gate": g["gate"]}
    rgb = [img[:3] + bg * T for _, img, T in planes]
    flat = torch.cat([c.reshape(-1) for c in rgb])
    if kind == "view":
        return {"rgb": flat, "T": torch.cat([T for _, _, T in planes])}
    if kind == "sweep":
        done = [c.view(3, v["height"], v["width"]) for c, v in zip(rgb, x["views"])]
        return done + [None] * (len(frames) - len(done))
    names = PARAM_KEYS
    if kind == "aux":
        (_, img, T), = planes
        up, ua = x["dL_drgb"].to(F64).view(3, -1), x["dL_daux"].to(F64).view(4, -1)
        g, _ = _adjoint(case, x, p, planes, [torch.cat([up, ua[:1], torch.zeros_like(ua[:2])])], [-ua[1]], names)
        aux = torch.cat([img[3:4], 1.0 - T[None], img[4:6]])
        return {"rgb": flat, "aux": aux.reshape(-1), "grads": [g[k] for k in names]}
    diff = flat - x["target"].to(F64)
    d_img, at, ups = diff.sign() / diff.numel(), 0, []
    for v in x["views"]:
        size = 3 * v["width"] * v["height"]
        ups.append(d_img[at:at + size].view(3, -1))
        at += size
    g, seen = _adjoint(case, x, p, planes, ups, [(u * bg).sum(0) for u in ups], names)
    loss = diff.abs().mean()
    if not case["mask"]:
        return {"rgb": flat, "loss": loss if case["autograd"] else loss[None], "grads": [g[k] for k in names]}
    M, sig = torch.sigmoid(p["mask_logit"]), torch.sigmoid(p["opacity_logit"])
    straight = (M * (1 - M)) * (g["log_scale"].sum(1) + g["opacity_logit"] / (1 - sig))
    stats = torch.zeros((case["n"], 4), dtype=F64, device=DEVICE)
    for rows, d_uv, d_mean in seen:
        stats[rows, 0] += d_uv.norm(dim=1)
        stats[rows, 1] += d_mean[rows, 3].abs()
        stats[rows, 2] += 1.0
    return {"mask_loss": M.mean()[None], "stats": stats, "rgb": flat, "loss": loss[None],
            "grads": [g[k] for k in names] + [straight + M * (1 - M) / case["n"]]}
