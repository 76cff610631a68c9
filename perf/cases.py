"""The work that users of this renderer have it do, as cases to be timed.

A case is a dict of plain values; `prepare` makes what a program has in hand
before the call (inputs from the seed, the Renderer or Server it keeps, the
buffers it reuses), `run` is one pass through the public entry points, `work`
the bytes and operations that pass cannot do without, `exact` its result in 64
bits from plain torch where that is feasible.

Kinds (the key "kind"):
  map       one mapping iteration: decode, render, weighted L1 loss with the
            mean-scale term, render backward, decode backward, all gradients
  autograd  the same path through the torch.autograd wrappers, the loss in torch
  plain     one plain-3DGS iteration (a Gaussian set, no decode)
  view      a rendered frame and its tracking uncertainty (no gradients)
  track     one tracking request served: three pyramid levels, pose gradient
  decode    the anchor decode alone; decode_bwd its backward alone
  lift      feature lifting and the distillation loss, all gradients
  ssim      the D-SSIM term and its gradient
  unc       the uncertainty MLP, its loss, mask and gradients
  anchors   the probabilistic anchor update on one keyframe

Sizes: 640x480 and 1280x720 frames and their ragged neighbours, 10k to 500k
anchors of 4 to 10 Gaussians, 0, 16 or 32 rendered feature channels.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2505_22335_gb300 import autograd as AG
from paper_2505_22335_gb300 import binding as B
from paper_2505_22335_gb300 import scenes

LAMBDA_SCALE = 0.01  # weight of the mean-scale term


def listed():
    return [
        # the smallest whole call: 2,000 plain Gaussians, one 160x120 view, RGB + depth
        dict(name="plain_2k_160x120", kind="plain", n=2000, V=1, W=160, H=120, NF=0),
        # a young map in a training script: 10k anchors, one frame, loss written in torch
        dict(name="autograd_10k_x10_640x480", kind="autograd", A=10_000, K=10, NF=16, V=1, W=640, H=480),
        # the mapping iteration of a grown map: 1M Gaussians, a batch of 8 keyframes
        dict(name="map_100k_x10_8x640x480", kind="map", A=100_000, K=10, NF=16, V=8, W=640, H=480, bf16=False),
        # the same on large frames with wide features and the tensor-core decode
        dict(name="map_100k_x10_8x1280x720_nf32", kind="map", A=100_000, K=10, NF=32, V=8, W=1280, H=720, bf16=True),
        # a viewer / tracking front end: one frame of a plain map at a ragged size, its residual and mask
        dict(name="view_300k_1237x693", kind="view", n=300_000, V=1, W=1237, H=693, NF=16),
        # camera-rate tracking against a resident map, through the server
        dict(name="track_500k_x10_640x480", kind="track", A=500_000, K=10, NF=16, W=640, H=480),
        # the decode alone, an odd anchor count and 3 keyframes
        dict(name="decode_61237_x10_3v", kind="decode", A=61_237, K=10, NF=16, V=3, bf16=False),
        # its backward alone (gradients of the MLPs, the anchors and the poses)
        dict(name="decode_bwd_40011_x10_4v", kind="decode_bwd", A=40_011, K=10, NF=16, V=4),
        # distillation against 384-wide DINO features for the keyframe batch
        dict(name="lift_8x640x480", kind="lift", NF=16, V=8, W=640, H=480, nh=384, patch=14),
        # the D-SSIM term for the keyframe batch
        dict(name="ssim_8x640x480", kind="ssim", V=8, W=640, H=480),
        # the uncertainty MLP for a batch of ragged frames
        dict(name="unc_5x621x467", kind="unc", V=5, W=621, H=467, nh=384, patch=14),
        # one keyframe entering the anchor map
        dict(name="anchors_100k_640x480", kind="anchors", A=100_000, K=10, W=640, H=480),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plain", "autograd", "map", "map", "view", "track", "decode", "decode_bwd", "lift", "ssim",
                       "unc", "anchors"])
    # frames from 160x120 to 1280x720, most of them not multiples of the tile
    W = _log(rng, 160, 1280)
    H = max(90, min(720, int(W * rng.uniform(0.55, 0.78))))
    V = rng.randint(1, 8)
    K = rng.choice([4, 8, 10])
    NF = rng.choice([0, 16, 16, 32])
    if kind == "plain":
        return dict(kind=kind, n=_log(rng, 1500, 300_000), V=rng.randint(1, 3), W=W, H=H, NF=NF)
    if kind == "autograd":
        return dict(kind=kind, A=_log(rng, 500, 50_000), K=K, NF=NF, V=rng.randint(1, 3), W=W, H=H)
    if kind == "map":
        return dict(kind=kind, A=_log(rng, 2000, 100_000), K=K, NF=NF, V=V, W=W, H=H, bf16=rng.random() < 0.4)
    if kind == "view":
        return dict(kind=kind, n=_log(rng, 5000, 500_000), V=rng.randint(1, 2), W=W, H=H, NF=NF)
    if kind == "track":
        return dict(kind=kind, A=_log(rng, 20_000, 500_000), K=K, NF=rng.choice([0, 16]), W=W // 4 * 4, H=H // 4 * 4)
    if kind == "decode":
        return dict(kind=kind, A=_log(rng, 1000, 150_000), K=K, NF=NF, V=rng.randint(1, 6), bf16=rng.random() < 0.3)
    if kind == "decode_bwd":
        return dict(kind=kind, A=_log(rng, 1000, 80_000), K=K, NF=NF, V=rng.randint(1, 6))
    if kind == "lift":
        return dict(kind=kind, NF=rng.choice([16, 16, 32]), V=rng.randint(1, 4), W=W, H=H,
                    nh=rng.choice([64, 384, 768]), patch=rng.choice([14, 16]))
    if kind == "ssim":
        return dict(kind=kind, V=V, W=W, H=H)
    if kind == "unc":
        return dict(kind=kind, V=rng.randint(1, 6), W=W, H=H, nh=rng.choice([64, 384, 768]),
                    patch=rng.choice([14, 14, 16]))
    return dict(kind=kind, A=_log(rng, 2000, 200_000), K=K, W=W, H=H)


# ---------------------------------------------------------------------------
# inputs (drawn on the GPU from the seed; distributions as in scenes.py)
# ---------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _u(g, *s, lo=0.0, hi=1.0):
    return torch.rand(*s, generator=g, device="cuda") * (hi - lo) + lo


def _n(g, *s, sigma=1.0):
    return torch.randn(*s, generator=g, device="cuda") * sigma


def _cams(c, seed, V=None):
    # 55 degrees or so across at every size, keyframes on the arc, odd temporal codes
    V = V or c.get("V", 1)
    cams = scenes.cameras(seed, V, c["W"], c["H"], 600.0 * c["W"] / 640.0)
    for i, cam in enumerate(cams):
        cam.t_norm = (i + 0.37) / (V + 1)
    return cams


def _plain(g, n, NF):
    centre = torch.tensor(scenes.CUBE_CENTRE, device="cuda", dtype=torch.float32)
    mean = centre + _u(g, n, 3, lo=-1.0, hi=1.0)
    # a map of more Gaussians has smaller ones
    hi = 0.05 * min(1.0, (20_000.0 / n) ** (1.0 / 3.0))
    scale = torch.exp(_u(g, n, 3, lo=math.log(0.1 * hi), hi=math.log(hi)))
    quat = torch.nn.functional.normalize(_n(g, n, 4), dim=1)
    z1 = torch.zeros(n, 1, device="cuda")
    op = torch.sigmoid(_n(g, n, 1))
    pack = lambda *t: torch.cat(t, 1).reshape(1, n, -1).contiguous()
    return B.GaussianSet(pack(mean, op), pack(scale, z1), pack(quat), pack(_u(g, n, 3), z1), _n(g, 1, n, NF), False)


def _anchors(g, A, K):
    centre = torch.tensor(scenes.CUBE_CENTRE, device="cuda", dtype=torch.float32)
    return dict(pos=(centre + _u(g, A, 3, lo=-1.0, hi=1.0)).contiguous(), feat=_n(g, A, 32, sigma=0.1),
                offsets=_n(g, A, K, 3, sigma=0.05),
                scaling=torch.exp(_u(g, A, 3, lo=math.log(0.01), hi=math.log(0.1))))


def _mlp(seed, K, NF):
    w = scenes.mlp_weights(seed + 1000, K, NF, bias_sigma=0.05)
    return {k: torch.tensor(v, dtype=torch.float32, device="cuda").contiguous() for k, v in w.items()}


def _targets(g, P, NF):
    return dict(color=_u(g, 3 * P), depth=_u(g, P, lo=1.5, hi=3.5), feat=_n(g, NF * P), weight=_u(g, P))


def _like(d):
    return {k: torch.zeros_like(v) for k, v in d.items()}


def _pixels(cams):
    return sum(c.width * c.height for c in cams)


def _lift_mlp(g, NF, nh):
    return dict(w1=_n(g, 128, NF, sigma=0.3), b1=_n(g, 128, sigma=0.1), w2=_n(g, nh, 128, sigma=0.1),
                b2=_n(g, nh, sigma=0.1))


def _patches(c):
    return -(-c["H"] // c["patch"]) * -(-c["W"] // c["patch"])


def _after_forward(R, cams, g, NF):
    """A small rendered set, so that the Renderer holds these views as its last forward's."""
    R.forward(_plain(g, 64, NF), cams)


def prepare(case, seed):
    c, kind, g = case, case["kind"], _gen(seed)
    s = dict(case=c)
    if kind in ("map", "autograd"):
        s["cams"] = _cams(c, seed)
        s["anc"], s["mlp"] = _anchors(g, c["A"], c["K"]), _mlp(seed, c["K"], c["NF"])
        P = _pixels(s["cams"])
        s["tgt"] = _targets(g, P, c["NF"])
        s["R"] = R = B.Renderer(n_feat=c["NF"], k=c["K"], decode_bf16=int(c.get("bf16", False)))
        if kind == "autograd":
            for t in (*s["anc"].values(), *s["mlp"].values()):
                t.requires_grad_(True)
            s["xi"] = torch.zeros(c["V"], 6, device="cuda", requires_grad=True)
            views, at = [], 0
            for cam in s["cams"]:
                h, w = cam.height, cam.width
                views.append(dict(color=s["tgt"]["color"][3 * at:3 * (at + h * w)].view(3, h, w),
                                  depth=s["tgt"]["depth"][at:at + h * w].view(h, w),
                                  feat=s["tgt"]["feat"][c["NF"] * at:c["NF"] * (at + h * w)].view(c["NF"], h, w),
                                  weight=s["tgt"]["weight"][at:at + h * w].view(h, w)))
                at += h * w
            s["views"] = views
        else:
            N = c["A"] * c["K"]
            s["g"], s["grad"] = (B.GaussianSet.empty(c["V"], N, c["NF"], True) for _ in range(2))
            s["img"] = R.alloc_images(s["cams"])
            s["loss"] = torch.zeros(1, device="cuda")
            s["dimg"] = _like({k: s["img"][k] for k in ("color", "depth", "feat")})
            s["d_pose"] = torch.zeros(c["V"], 6, device="cuda")
            s["d_mlp"], s["d_anc"] = _like(s["mlp"]), _like(s["anc"])
    elif kind in ("plain", "view"):
        s["cams"] = _cams(c, seed)
        s["g"] = _plain(g, c["n"], c["NF"])
        s["tgt"] = _targets(g, _pixels(s["cams"]), c["NF"])
        s["R"] = R = B.Renderer(n_feat=c["NF"])
        s["img"] = R.alloc_images(s["cams"])
        if kind == "plain":
            s["dimg"] = _like({k: s["img"][k] for k in ("color", "depth", "feat")})
            s["loss"] = torch.zeros(1, device="cuda")
            s["grad"] = B.GaussianSet.empty(1, c["n"], c["NF"], False)
            s["d_pose"] = torch.zeros(c["V"], 6, device="cuda")
    elif kind == "track":
        s["anc"], s["mlp"] = _anchors(g, c["A"], c["K"]), _mlp(seed, c["K"], c["NF"])
        s["cams"] = _cams(c, seed, 1)
        P = sum((c["W"] >> l) * (c["H"] >> l) for l in range(3))
        s["tgt"] = _targets(g, P, c["NF"])
        s["loss"], s["d_pose"] = torch.zeros(1, device="cuda"), torch.zeros(6, device="cuda")
        torch.cuda.synchronize()  # the server's streams read what was made on this one
        s["srv"] = B.Server(s["anc"], s["mlp"], n_feat=c["NF"], k=c["K"], slots=1, decode_bf16=1)
    elif kind in ("decode", "decode_bwd"):
        s["cams"] = _cams(dict(c, W=640, H=480), seed)
        s["anc"], s["mlp"] = _anchors(g, c["A"], c["K"]), _mlp(seed, c["K"], c["NF"])
        s["R"] = B.Renderer(n_feat=c["NF"], k=c["K"], decode_bf16=int(c.get("bf16", False)))
        V, N = c["V"], c["A"] * c["K"]
        s["g"] = B.GaussianSet.empty(V, N, c["NF"], True)
        if kind == "decode_bwd":
            for k in ("mean_opacity", "scale", "quat", "color", "feat"):
                t = getattr(s["g"], k)
                t.copy_(_n(g, *t.shape))
            s["d_mlp"], s["d_anc"] = _like(s["mlp"]), _like(s["anc"])
            s["d_pose"] = torch.zeros(V, 6, device="cuda")
    elif kind == "lift":
        s["cams"] = _cams(c, seed)
        P = _pixels(s["cams"])
        s["feat"], s["weight"] = _n(g, c["NF"] * P), _u(g, P)
        s["dino"] = _n(g, c["V"] * _patches(c) * c["nh"])
        s["mlp"] = _lift_mlp(g, c["NF"], c["nh"])
        s["R"] = B.Renderer(n_feat=c["NF"])
        _after_forward(s["R"], s["cams"], g, c["NF"])
        s["d_mlp"], s["d_feat"] = _like(s["mlp"]), torch.zeros_like(s["feat"])
        s["loss"] = torch.zeros(1, device="cuda")
    elif kind == "ssim":
        s["cams"] = _cams(c, seed)
        P = _pixels(s["cams"])
        # photographs, and renders a little off them: smooth structure plus noise
        base, at = [], 0
        for cam in s["cams"]:
            low = _u(g, 1, 3, 12, 16)
            base.append(torch.nn.functional.interpolate(low, size=(cam.height, cam.width), mode="bilinear",
                                                        align_corners=False).reshape(-1))
        base = torch.cat(base)
        s["target"] = (base + _n(g, 3 * P, sigma=0.03)).clamp(0, 1).contiguous()
        s["color"] = (base + _n(g, 3 * P, sigma=0.05)).clamp(0, 1).contiguous()
        s["weight"] = (_u(g, P) > 0.1).float()
        s["R"] = B.Renderer(n_feat=0)
        _after_forward(s["R"], s["cams"], g, 0)
        s["d_color"], s["loss"] = torch.zeros_like(s["color"]), torch.zeros(1, device="cuda")
    elif kind == "unc":
        s["cams"] = _cams(c, seed)
        P = _pixels(s["cams"])
        s["dino"], s["Rmap"] = _n(g, c["V"] * _patches(c) * c["nh"]), _u(g, P)
        s["mlp"] = dict(w1=_n(g, 128, c["nh"], sigma=1.96 / math.sqrt(c["nh"])), b1=_n(g, 128, sigma=0.1),
                        w2=_n(g, 128, sigma=0.1), b2=torch.full((1,), 0.2, device="cuda"))
        s["R"] = B.Renderer(n_feat=0)
        _after_forward(s["R"], s["cams"], g, 0)
        s["d_mlp"], s["loss"] = _like(s["mlp"]), torch.zeros(1, device="cuda")
        s["out"] = dict(sigma=torch.empty(P, device="cuda"), motion=torch.empty(P, dtype=torch.uint8, device="cuda"))
    elif kind == "anchors":
        # the keyframe and the anchors' places go by the case, so that the map grows to the same size
        # for every seed; their order in the arrays, features, offsets and scalings by the seed
        s["cams"] = _cams(c, c["A"], 1)
        depth, motion = scenes.keyframe(c["A"] + 1, s["cams"][0])
        anc, logodds = scenes.anchor_cloud(c["A"] + 2, s["cams"][0], depth, c["A"], c["K"])
        t = lambda a, dt=torch.float32: torch.tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")
        order = torch.randperm(c["A"], generator=g, device="cuda")
        s["anc"] = dict(_anchors(g, c["A"], c["K"]), pos=t(anc["pos"])[order].contiguous())
        s["logodds"] = t(logodds)[order].contiguous()
        s["depth"], s["motion"] = t(depth), t(motion, torch.uint8)
        s["R"] = B.Renderer(k=c["K"])
    else:
        raise ValueError(kind)
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _zero(d):
    for v in d.values():
        v.zero_()


def _run_map(s):
    c, R = s["case"], s["R"]
    R.decode(s["anc"], s["mlp"], s["cams"], out=s["g"])
    R.forward(s["g"], s["cams"], out=s["img"])
    R.loss(s["img"], s["tgt"], lambda_scale=LAMBDA_SCALE, g=s["g"], loss_out=s["loss"], grad_out=s["dimg"])
    R.backward(s["dimg"], B.GRAD_ALL, scale_grad=LAMBDA_SCALE / (3.0 * c["V"] * c["A"] * c["K"]), grad=s["grad"],
               d_pose=s["d_pose"])
    _zero(s["d_mlp"])
    _zero(s["d_anc"])
    R.decode_backward(s["anc"], s["mlp"], s["cams"], s["grad"], B.GRAD_ALL, s["d_mlp"], s["d_anc"], s["d_pose"])
    return dict(loss=s["loss"], img=s["img"], d_pose=s["d_pose"], d_mlp=s["d_mlp"], d_anc=s["d_anc"])


def _run_autograd(s):
    leaves = [*s["anc"].values(), *s["mlp"].values(), s["xi"]]
    for t in leaves:
        t.grad = None
    outs, _ = AG.render_anchors(s["R"], s["cams"], s["anc"], s["mlp"], s["xi"])
    loss = 0.0
    for o, t in zip(outs, s["views"]):
        w = t["weight"]
        term = (w * (o["color"] - t["color"]).abs().sum(0)).mean() + (w * (o["depth"] - t["depth"]).abs()).mean()
        if s["case"]["NF"]:
            term = term + (w * (o["feat"] - t["feat"]).abs().sum(0)).mean()
        loss = loss + term / len(outs)
    loss.backward()
    return dict(loss=loss.detach(), color=[o["color"].detach() for o in outs],
                depth=[o["depth"].detach() for o in outs], grads=[t.grad for t in leaves])


def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "map":
        return _run_map(s)
    if kind == "autograd":
        return _run_autograd(s)
    R = s.get("R")
    if kind == "plain":
        R.forward(s["g"], s["cams"], out=s["img"])
        R.loss(s["img"], s["tgt"], loss_out=s["loss"], grad_out=s["dimg"])
        R.backward(s["dimg"], B.GRAD_POSE | B.GRAD_GAUSS, grad=s["grad"], d_pose=s["d_pose"])
        d = s["grad"]
        return dict(loss=s["loss"], img=s["img"], d_pose=s["d_pose"], d_mean_opacity=d.mean_opacity, d_scale=d.scale,
                    d_quat=d.quat, d_color=d.color, d_feat=d.feat)
    if kind == "view":
        R.forward(s["g"], s["cams"], out=s["img"])
        return dict(img=s["img"], unc=R.tracking_uncertainty(s["img"], s["tgt"]))
    if kind == "track":
        srv = s["srv"]
        srv.wait(srv.submit(B.TRACK, s["cams"], s["tgt"], s["loss"], s["d_pose"], levels=3))
        return dict(loss=s["loss"], d_pose=s["d_pose"])
    if kind == "decode":
        g = R.decode(s["anc"], s["mlp"], s["cams"], out=s["g"])
        return dict(mean_opacity=g.mean_opacity, scale=g.scale, quat=g.quat, color=g.color, feat=g.feat)
    if kind == "decode_bwd":
        _zero(s["d_mlp"])
        _zero(s["d_anc"])
        s["d_pose"].zero_()
        R.decode_backward(s["anc"], s["mlp"], s["cams"], s["g"], B.GRAD_ALL, s["d_mlp"], s["d_anc"], s["d_pose"])
        return dict(d_mlp=s["d_mlp"], d_anc=s["d_anc"], d_pose=s["d_pose"])
    if kind == "lift":
        _zero(s["d_mlp"])
        s["d_feat"].zero_()
        R.feature_lift(s["feat"], s["dino"], s["mlp"], n_h=c["nh"], patch=c["patch"], scale=0.4, d_mlp=s["d_mlp"],
                       d_feat=s["d_feat"], weight=s["weight"], loss_out=s["loss"])
        return dict(loss=s["loss"], d_mlp=s["d_mlp"], d_feat=s["d_feat"])
    if kind == "ssim":
        s["d_color"].zero_()
        R.ssim_loss(s["color"], s["target"], scale=0.2, d_color=s["d_color"], weight=s["weight"], loss_out=s["loss"])
        return dict(loss=s["loss"], d_color=s["d_color"])
    if kind == "unc":
        _zero(s["d_mlp"])
        R.uncertainty_mlp(s["dino"], s["Rmap"], s["mlp"], n_h=c["nh"], patch=c["patch"], d_mlp=s["d_mlp"],
                          out=s["out"], loss_out=s["loss"])
        return dict(loss=s["loss"], d_mlp=s["d_mlp"], sigma=s["out"]["sigma"], motion=s["out"]["motion"])
    if kind == "anchors":
        anc, logodds, src, counts = R.anchor_update(s["anc"], s["logodds"], s["cams"][0], s["depth"], s["motion"],
                                                    capacity=2 * c["A"])
        return dict(anc=anc, logodds=logodds, src=src, counts=counts)
    raise ValueError(kind)


# ---------------------------------------------------------------------------
# what one pass cannot do without
# ---------------------------------------------------------------------------

def _decode_flops(rows, K, NF, back):
    fwd = 2 * (38 * 128 + 32 * K * (11 + NF))
    # recomputed hidden layer and non-linear outputs, dL/dH, dL/dx, and both weight gradients
    bwd = 2 * (38 * 128 + 7 * K * 32 + 32 * K * (11 + NF) + 36 * 128) + 2 * (32 * K * (11 + NF) + 128 * 39)
    return rows * (bwd if back else fwd)


# (pixel, Gaussian) pairs blended until a pixel is opaque, about what these scenes show
PAIRS = 100


def work(case):
    c, kind = case, case["kind"]
    P = c.get("V", 1) * c.get("W", 640) * c.get("H", 480)
    NF = c.get("NF", 0)
    img_b = 4 * P * (6 + NF)            # images written (colour, depth, T, n_contrib, features)
    tgt_b = 4 * P * (5 + NF)            # targets and weights read
    fwd_pair, bwd_pair = 2 * (NF + 4) + 12, 4 * NF + 60
    if kind in ("map", "autograd", "track", "decode", "decode_bwd"):
        A, K, V = c["A"], c["K"], c.get("V", 1)
        anc_b = 4 * A * (3 + 32 + 3 * K + 3)
        set_b = 4 * V * A * K * (16 + NF)
        rows = A * V
    if kind in ("map", "autograd"):
        return dict(bytes=2 * anc_b + tgt_b + img_b, flops=_decode_flops(rows, K, NF, False) +
                    _decode_flops(rows, K, NF, True) + P * PAIRS * (fwd_pair + bwd_pair))
    if kind == "track":
        P = P * 21 // 16
        return dict(bytes=anc_b + 4 * P * (5 + NF), flops=_decode_flops(rows, K, NF, False) +
                    P * PAIRS * (fwd_pair + bwd_pair))
    if kind == "decode":
        return dict(bytes=anc_b + set_b, flops=_decode_flops(rows, K, NF, False))
    if kind == "decode_bwd":
        return dict(bytes=2 * anc_b + set_b, flops=_decode_flops(rows, K, NF, True))
    if kind in ("plain", "view"):
        n_b = 4 * c["n"] * (16 + NF)
        if kind == "view":
            return dict(bytes=n_b + img_b + 4 * P * (4 + NF) + 9 * P, flops=P * PAIRS * fwd_pair)
        return dict(bytes=2 * n_b + img_b + tgt_b, flops=P * PAIRS * (fwd_pair + bwd_pair))
    if kind == "lift":
        np_ = c["V"] * _patches(c)
        # the gradients without the nh-wide map: first layer and its two products, two 128 x 128 products
        return dict(bytes=4 * P * (2 * NF + 1) + 4 * np_ * c["nh"],
                    flops=P * (6 * NF * 128 + 4 * 128 * 128 + 28 * 128) + np_ * 4 * 128 * c["nh"])
    if kind == "ssim":
        # two images read, the gradient written, the weights read; separable 11-tap windows of 5 + 3 maps
        return dict(bytes=4 * 3 * P * 3 + 4 * P, flops=3 * P * (8 * 2 * 11 * 2 + 60))
    if kind == "unc":
        np_ = c["V"] * _patches(c)
        return dict(bytes=4 * np_ * c["nh"] + 9 * P, flops=P * 22 * 128 + np_ * 4 * 128 * c["nh"])
    if kind == "anchors":
        row = 4 * (3 + 32 + 3 * c["K"] + 3 + 1)
        return dict(bytes=2 * c["A"] * row + 5 * P, flops=60 * (c["A"] + P))
    raise ValueError(kind)


# ---------------------------------------------------------------------------
# the results in 64 bits, in plain torch
# ---------------------------------------------------------------------------

def _exact_decode(anc, mlp, cams, K, NF, xi=None):
    """Decoded sets [V, A K, .] in 64 bits; xi [V, 6]: pose twists (the camera centre moves)."""
    A = anc["pos"].shape[0]
    outs = dict(mean_opacity=[], scale=[], quat=[], color=[], feat=[])
    zero = torch.zeros(A * K, 1, dtype=torch.float64, device="cuda")
    for v, cam in enumerate(cams):
        T = torch.tensor(np.float32(cam.T_cw).astype(np.float64), device="cuda")
        Rm, t = T[:3, :3], T[:3, 3]
        oc = -(Rm.T @ t)
        if xi is not None:
            # Exp(xi) T: the centre -R^T t moves by -R^T rho to first order (phi leaves it in place)
            oc = oc - Rm.T @ xi[v, :3]
        r = anc["pos"] - oc
        d = r.norm(dim=1, keepdim=True)
        tn = float(np.float32(cam.t_norm)) * math.pi
        enc = torch.tensor([math.sin(tn), math.cos(tn)], dtype=torch.float64, device="cuda").expand(A, 2)
        x = torch.cat([anc["feat"], r / d, d, enc], 1)
        z = x @ mlp["w1"].T + mlp["b1"]
        h = [torch.relu(z[:, :32]), torch.relu(z[:, 32:64]), torch.relu(z[:, 64:96]),
             torch.nn.functional.softplus(z[:, 96:], threshold=50.0)]
        lo = [0, K, 8 * K, 11 * K, K * (11 + NF)]
        y = [h[i] @ mlp["w2"][lo[i]:lo[i + 1]].T + mlp["b2"][lo[i]:lo[i + 1]] for i in range(4)]
        mean = (anc["pos"][:, None, :] + anc["offsets"]).reshape(A * K, 3)
        cov = y[1].reshape(A, K, 7)
        outs["mean_opacity"].append(torch.cat([mean, torch.sigmoid(y[0]).reshape(A * K, 1)], 1))
        outs["scale"].append(torch.cat([(anc["scaling"][:, None, :] * torch.sigmoid(cov[..., :3])).reshape(-1, 3),
                                        zero], 1))
        outs["quat"].append(cov[..., 3:].reshape(-1, 4))
        outs["color"].append(torch.cat([torch.sigmoid(y[2]).reshape(-1, 3), zero], 1))
        outs["feat"].append(y[3].reshape(A * K, NF))
    return {k: torch.stack(v) for k, v in outs.items()}


def _f64(d):
    return {k: v.double() for k, v in d.items()}


def _exact_decode_bwd(s):
    c = s["case"]
    G = {k: getattr(s["g"], k).double() for k in ("mean_opacity", "scale", "quat", "color", "feat")}
    mlp = {k: v.requires_grad_(True) for k, v in _f64(s["mlp"]).items()}
    d_anc = {k: [] for k in s["anc"]}
    xi = torch.zeros(c["V"], 6, dtype=torch.float64, device="cuda", requires_grad=True)
    A, K, step = c["A"], c["K"], 20_000
    for a in range(0, A, step):  # by anchors: the rows are independent
        anc = {k: v[a:a + step].double().requires_grad_(True) for k, v in s["anc"].items()}
        o = _exact_decode(anc, mlp, s["cams"], K, c["NF"], xi)
        sum((o[k] * G[k][:, a * K:(a + step) * K]).sum() for k in G).backward()
        for k in d_anc:
            d_anc[k].append(anc[k].grad)
    return dict(d_mlp={k: v.grad for k, v in mlp.items()}, d_anc={k: torch.cat(v) for k, v in d_anc.items()},
                d_pose=xi.grad)


def _window():
    k = torch.arange(-5, 6, dtype=torch.float64, device="cuda")
    w = torch.exp(-k * k / (2 * 1.5 ** 2))
    return w / w.sum()


def _blur(t):
    w, ch = _window(), t.shape[1]
    f = torch.nn.functional.conv2d
    t = f(t, w.view(1, 1, 1, 11).expand(ch, 1, 1, 11), padding=(0, 5), groups=ch)
    return f(t, w.view(1, 1, 11, 1).expand(ch, 1, 11, 1), padding=(5, 0), groups=ch)


def _exact_ssim(s):
    P, at, loss, grads = _pixels(s["cams"]), 0, 0.0, []
    for cam in s["cams"]:
        h, w = cam.height, cam.width
        cut = lambda t, ch: t[ch * at:ch * (at + h * w)].double().view(1, ch, h, w)
        x, y, m = cut(s["color"], 3).clone().requires_grad_(True), cut(s["target"], 3), cut(s["weight"], 1)
        mx, my = _blur(x), _blur(y)
        A1, A2 = 2 * mx * my + 1e-4, 2 * (_blur(x * y) - mx * my) + 9e-4
        B1, B2 = mx * mx + my * my + 1e-4, _blur(x * x) - mx * mx + _blur(y * y) - my * my + 9e-4
        part = 0.2 * (m * (1 - A1 * A2 / (B1 * B2))).sum() / (3 * P)
        part.backward()
        loss += part.detach()
        grads.append(x.grad.reshape(-1))
        at += h * w
    return dict(loss=loss.reshape(1), d_color=torch.cat(grads))


def _upsample(grid, c, rows):
    """DINO features of image rows `rows` (a slice) of one view: [rows, W, nh] in 64 bits."""
    hp, wp, p = -(-c["H"] // c["patch"]), -(-c["W"] // c["patch"]), c["patch"]
    grid = grid.double().view(hp, wp, c["nh"])

    def axis(n, np_):
        u = ((torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) / p - 0.5).clamp(0, np_ - 1)
        i = u.floor().long()
        return i, (i + 1).clamp(max=np_ - 1), u - i
    y0, y1, fy = (t[rows] for t in axis(c["H"], hp))
    x0, x1, fx = axis(c["W"], wp)
    fy, fx = fy.view(-1, 1, 1), fx.view(1, -1, 1)
    at = lambda y, x: grid[y][:, x]
    return (1 - fy) * ((1 - fx) * at(y0, x0) + fx * at(y0, x1)) + fy * ((1 - fx) * at(y1, x0) + fx * at(y1, x1))


def _per_rows(s, rows=64):
    """(view index, pixel offset, row slice) in blocks of image rows."""
    at = 0
    for v, cam in enumerate(s["cams"]):
        for r in range(0, cam.height, rows):
            yield v, at, slice(r, min(cam.height, r + rows))
        at += cam.height * cam.width


def _exact_lift(s):
    c = s["case"]
    P, W, H, NF, n = _pixels(s["cams"]), c["W"], c["H"], c["NF"], _patches(c) * c["nh"]
    mlp = {k: v.requires_grad_(True) for k, v in _f64(s["mlp"]).items()}
    feat = s["feat"].double()
    d_feat, loss = torch.zeros_like(feat), 0.0
    for v, at, rows in _per_rows(s):
        F = _upsample(s["dino"][v * n:(v + 1) * n], c, rows).reshape(-1, c["nh"])
        x = feat[NF * at:NF * (at + H * W)].view(NF, H, W)[:, rows].reshape(NF, -1).T.clone().requires_grad_(True)
        w = s["weight"][at:at + H * W].view(H, W)[rows].reshape(-1).double()
        Fh = torch.relu(x @ mlp["w1"].T + mlp["b1"]) @ mlp["w2"].T + mlp["b2"]
        part = 0.4 * (w * (1 - torch.nn.functional.cosine_similarity(F, Fh, dim=1, eps=1e-30))).sum() / P
        part.backward()
        loss += part.detach()
        d_feat[NF * at:NF * (at + H * W)].view(NF, H, W)[:, rows] = x.grad.T.reshape(NF, -1, W)
    return dict(loss=loss.reshape(1), d_mlp={k: v.grad for k, v in mlp.items()}, d_feat=d_feat)


def _exact_unc(s):
    c = s["case"]
    P, W, H, n = _pixels(s["cams"]), c["W"], c["H"], _patches(c) * c["nh"]
    mlp = {k: v.requires_grad_(True) for k, v in _f64(s["mlp"]).items()}
    sigma, loss = [], 0.0
    for v, at, rows in _per_rows(s):
        F = _upsample(s["dino"][v * n:(v + 1) * n], c, rows).reshape(-1, c["nh"])
        R = s["Rmap"][at:at + H * W].view(H, W)[rows].reshape(-1).double()
        z = torch.relu(F @ mlp["w1"].T + mlp["b1"]) @ mlp["w2"] + mlp["b2"]
        sg = torch.nn.functional.softplus(z, threshold=50.0)
        part = (R / (2 * sg * sg) + torch.log(sg)).sum() / P
        part.backward()
        loss += part.detach()
        sigma.append(sg.detach())
    return dict(loss=loss.reshape(1), d_mlp={k: v.grad for k, v in mlp.items()}, sigma=torch.cat(sigma), motion=None)


def _exact_plain(s):
    """Brute force over all (pixel, Gaussian) pairs of a small plain scene, gradients by autograd."""
    c = s["case"]
    if c["V"] != 1 or c["n"] * c["W"] * c["H"] > 60_000_000:
        return None
    amin, amax, tmin = float(np.float32(1.0 / 255.0)), float(np.float32(0.99)), float(np.float32(1e-4))
    cam, NF, W, H = s["cams"][0], c["NF"], c["W"], c["H"]
    leaf = {k: getattr(s["g"], k)[0].double().requires_grad_(True)
            for k in ("mean_opacity", "scale", "quat", "color", "feat")}
    xi = torch.zeros(6, dtype=torch.float64, device="cuda", requires_grad=True)
    T = torch.tensor(np.float32(cam.T_cw).astype(np.float64), device="cuda")
    K = torch.zeros(3, 3, dtype=torch.float64, device="cuda")
    skew = K.index_put((torch.tensor([2, 0, 1], device="cuda"), torch.tensor([1, 2, 0], device="cuda")), xi[3:]) \
        - K.index_put((torch.tensor([1, 2, 0], device="cuda"), torch.tensor([2, 0, 1], device="cuda")), xi[3:])
    Rot = T[:3, :3] + skew @ T[:3, :3]
    t = T[:3, 3] + skew @ T[:3, 3] + xi[:3]
    mean, op = leaf["mean_opacity"][:, :3], leaf["mean_opacity"][:, 3]
    p = mean @ Rot.T + t
    X, Y, Z = p.unbind(1)
    ok = (Z > 0.2) & ((X / Z).abs() <= 1.3 * 0.5 * W / cam.fx) & ((Y / Z).abs() <= 1.3 * 0.5 * H / cam.fy) & (op >= amin)
    order = torch.argsort(Z.detach().float().double(), stable=True)
    order = order[ok[order]]
    q = torch.nn.functional.normalize(leaf["quat"], dim=1)
    w, x, y, z = q.unbind(1)
    R = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y), 2 * (x * y + w * z),
                     1 - 2 * (x * x + z * z), 2 * (y * z - w * x), 2 * (x * z - w * y), 2 * (y * z + w * x),
                     1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    M = R * leaf["scale"][:, None, :3]
    o = torch.zeros_like(Z)
    J = torch.stack([cam.fx / Z, o, -cam.fx * X / Z ** 2, o, cam.fy / Z, -cam.fy * Y / Z ** 2], 1).view(-1, 2, 3)
    S = (J @ Rot) @ (M @ M.transpose(1, 2)) @ (J @ Rot).transpose(1, 2)
    a_, b_, c_ = S[:, 0, 0] + float(np.float32(0.3)), S[:, 0, 1], S[:, 1, 1] + float(np.float32(0.3))
    det = a_ * c_ - b_ * b_
    ii = torch.arange(W, dtype=torch.float64, device="cuda").repeat(H)
    jj = torch.arange(H, dtype=torch.float64, device="cuda").repeat_interleave(W)
    cut = lambda t: t[order][:, None]
    dx, dy = ii - cut(cam.fx * X / Z + cam.cx), jj - cut(cam.fy * Y / Z + cam.cy)
    power = -0.5 * (cut(c_ / det) * dx * dx - 2 * cut(b_ / det) * dx * dy + cut(a_ / det) * dy * dy)
    alpha = (cut(op) * torch.exp(power)).clamp(max=amax)
    alpha = torch.where(alpha >= amin, alpha, torch.zeros_like(alpha))
    after = torch.cumprod(1 - alpha, 0)
    before = torch.cat([torch.ones_like(after[:1]), after[:-1]])
    wgt = torch.where(after >= tmin, alpha * before, torch.zeros_like(alpha))
    Tf = torch.where(after >= tmin, after, torch.ones_like(after)).min(0).values
    color, depth = (wgt.T @ leaf["color"][order][:, :3]).T, wgt.T @ Z[order]
    feat = (wgt.T @ leaf["feat"][order]).T
    tg = _f64(s["tgt"])
    P = W * H
    loss = (tg["weight"] * ((color - tg["color"].view(3, P)).abs().sum(0) + (depth - tg["depth"]).abs() +
                            (feat - tg["feat"].view(NF, P)).abs().sum(0))).sum() / P
    grads = torch.autograd.grad(loss, [*leaf.values(), xi], allow_unused=True)
    gr = {k: (torch.zeros_like(v) if d is None else d).unsqueeze(0) for (k, v), d in zip(leaf.items(), grads)}
    return dict(loss=loss.detach().reshape(1), d_pose=grads[-1].reshape(1, 6),
                img=dict(color=color.detach().reshape(-1), depth=depth.detach(), feat=feat.detach().reshape(-1),
                         T=Tf.detach(), n_contrib=None),
                d_mean_opacity=gr["mean_opacity"], d_scale=gr["scale"], d_quat=gr["quat"], d_color=gr["color"],
                d_feat=gr["feat"])


def exact(case, seed):
    """Results in 64 bits; None for whole renders of large scenes (hours in plain torch) and for the
    anchor update (decisions and copies in float32, nothing computed beyond one addition)."""
    kind = case["kind"]
    if kind not in ("decode", "decode_bwd", "lift", "ssim", "unc", "plain"):
        return None
    s = prepare(case, seed)
    if kind == "decode":
        with torch.no_grad():
            return _exact_decode(_f64(s["anc"]), _f64(s["mlp"]), s["cams"], case["K"], case["NF"])
    return dict(decode_bwd=_exact_decode_bwd, lift=_exact_lift, ssim=_exact_ssim, unc=_exact_unc,
                plain=_exact_plain)[kind](s)
