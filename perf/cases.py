"""The workloads whose speed matters to a user of this framework, through its public entry points.

Each case is one call (or one training step) of Multi-Scale Deformable Aggregation as a program around it makes it:

* ``forward``  msda.forward: a decoder layer's feature aggregation at inference;
* ``serve``    msda.keypoints, then msda.forward on its locations: anchors to features, per decoder layer;
* ``oae``      msda.forward_oae: the aggregation with the visibility-weighted fusion over cameras;
* ``train``    the differentiable msda.msda and its (deterministic) gradients by torch.autograd;
* ``step``     msda.forward and the deterministic msda.backward into buffers that the caller keeps;
* ``atomic``   msda.forward_train and the atomic msda.backward into buffers that the caller keeps;
* ``batched``  msda.plan_batched(...).run(): many scenes of uneven size in one persistent launch.

Sampling locations are either ``uniform`` over the image and a margin, with a share of the (anchor, camera) pairs
out of view, or ``projected``: the keypoints of boxes on a floor seen by a ring of cameras, so that the keypoints of
an anchor fall close together and an anchor is in view of some cameras only.  Inputs are drawn on the GPU.
"""
import math
import random

import torch

from paper_2601_10819_gb300 import inputs, msda

_DT = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
_BASE = dict(kind="forward", B=1, cams=6, A=900, P=13, C=256, G=8, feat="bf16", w="bf16", height=540, width=960,
             stride=8, scales=4, mixed=False, loc="uniform", margin=0.0, away=0.0)


def _case(name=None, **kw):
    c = dict(_BASE, **kw)
    if name:
        c["name"] = name
    return c


_SPARSE4D = dict(height=256, width=704, stride=4, margin=0.05)  # a 256x704 image at strides 4..32


def listed():
    return [
        # the smallest call there is in earnest: a toy model, a unit test, one gradient check; launches and host work
        _case("tiny-forward-f32", cams=2, A=16, P=4, C=32, G=4, feat="f32", w="f32", height=16, width=16, stride=1,
              scales=2, margin=0.1),
        _case("tiny-train-f32", kind="train", cams=2, A=16, P=4, C=32, G=4, feat="f32", w="f32", height=16, width=16,
              stride=1, scales=2, margin=0.1),
        # one decoder layer of a six-camera vehicle model at inference, in FP32
        _case("sparse4d-6cam-forward-f32", feat="f32", w="f32", **_SPARSE4D),
        # the same with the keypoint projection in front, in BF16: what a serving loop runs per layer
        _case("sparse4d-6cam-serve-bf16", kind="serve", **dict(_SPARSE4D, loc="projected", margin=0.0)),
        # one decoder layer of an outside-in model over 64 cameras, 40 % of the (anchor, camera) pairs out of view
        _case("outside-in-64cam-forward-bf16", cams=64, away=0.4),
        # the occlusion-aware fusion over the cameras of one hall, FP16 as an inference engine has it
        _case("outside-in-24cam-oae-f16", kind="oae", cams=24, feat="f16", w="f16", height=360, width=640,
              loc="projected"),
        # a training step on the 64-camera frame into buffers that the training loop keeps
        _case("outside-in-64cam-step-bf16", kind="step", cams=64, away=0.4),
        # the training step of a 16-camera model, batch 4, through autograd: BF16 features, FP32 weights
        _case("train-16cam-b4-bf16", kind="train", B=4, cams=16, w="f32", **_SPARSE4D),
        # the same model trained with the atomic gradient (not reproducible), batch 2
        _case("train-16cam-b2-atomic-bf16", kind="atomic", B=2, cams=16, w="f32", **_SPARSE4D),
        # training on projected keypoints: anchors crowd the cells that the floor projects to
        _case("outside-in-20cam-train-projected-bf16", kind="train", cams=20, loc="projected"),
        # odd sizes, two resolutions among the cameras, three scales, FP32: a small model of one's own
        _case("ragged-5cam-train-f32", kind="train", B=2, cams=5, A=333, P=7, C=128, G=4, feat="f32", w="f32",
              height=203, width=331, stride=4, scales=3, mixed=True, margin=0.05, away=0.2),
        # serving 16 sites from one GPU: 4 to 96 cameras each, 720p and 1080p, 600 to 1200 anchors
        _case("batched-16-scenes-bf16", kind="batched", cams=96, A=1200, away=0.4, scenes=16, sizes=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward", "forward", "serve", "oae", "train", "train", "step", "atomic", "batched"])
    C, G = rng.choice([(32, 4), (64, 4), (64, 8), (128, 4), (128, 8), (256, 4), (256, 8), (256, 8), (256, 16)])
    ft, wt = rng.choice([("f32", "f32"), ("bf16", "bf16"), ("bf16", "bf16"), ("bf16", "f32"), ("f16", "f16")])
    loc = "projected" if kind == "serve" else rng.choice(["uniform", "projected"])
    c = _case(kind=kind, B=1 if kind in ("batched", "oae") else rng.choice([1, 1, 2, 3, 4]), cams=_log(rng, 1, 64),
              A=_log(rng, 16, 1200), P=rng.randint(1, 13), C=C, G=G, feat=ft, w=wt, height=rng.randint(16, 640),
              width=rng.randint(16, 960), stride=rng.choice([4, 8]), scales=rng.randint(1, 4),
              mixed=rng.random() < 0.4, loc=loc, margin=0.0 if loc == "projected" else rng.choice([0.0, 0.05, 0.1]),
              away=0.0 if loc == "projected" else rng.choice([0.0, 0.2, 0.4]))
    if kind == "batched":
        c.update(loc="uniform", scenes=rng.randint(2, 16), sizes=rng.randint(0, 10 ** 6))
    # no dearer than the largest listed cases: at most as many samples, and as many feature channels, as they have
    most = 1_500_000 if kind in ("train", "step", "atomic") else 3_000_000
    while c["B"] * c["cams"] * c["A"] * c["P"] * c["scales"] * c.get("scenes", 1) * c["C"] > most * 256:
        if c["cams"] > 1:
            c["cams"] = max(1, c["cams"] * 2 // 3)
        else:
            c["A"] = max(16, c["A"] * 2 // 3)
    while c["B"] * c["C"] * c.get("scenes", 1) * sum(h * w for m in _cam_maps(c) for h, w in m) > 360_000_000:
        c["height"], c["width"] = max(16, c["height"] * 4 // 5), max(16, c["width"] * 4 // 5)
        if c["height"] == 16 and c["width"] == 16:
            break
    return c


# ---------------------------------------------------------------------------
# Shapes
# ---------------------------------------------------------------------------
def _maps(height, width, c):
    strides = [c["stride"] << s for s in range(c["scales"])]
    return [(math.ceil(height / s), math.ceil(width / s)) for s in strides]


def _cam_maps(c):
    """Map sizes per camera; with ``mixed`` every third camera has two thirds of the resolution."""
    full, less = _maps(c["height"], c["width"], c), _maps(c["height"] * 2 // 3, c["width"] * 2 // 3, c)
    return [less if c["mixed"] and k % 3 == 2 else full for k in range(c["cams"])]


def _scenes(c):
    """The scenes of a batched case, each as a case of its own."""
    if c["kind"] != "batched":
        return [c]
    r = random.Random(c["sizes"])
    got = []
    for _ in range(c["scenes"]):
        small = r.random() < 0.5
        got.append(dict(c, cams=r.randint(min(4, c["cams"]), c["cams"]), A=r.randint(max(1, c["A"] // 2), c["A"]),
                        height=c["height"] * 2 // 3 if small else c["height"],
                        width=c["width"] * 2 // 3 if small else c["width"]))
    return got


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _project(anchors, offsets, dt, proj, img_wh):
    """Keypoints of the boxes moved by their velocity, seen by each camera: [B, A, P, K, 2] in the inputs' type."""
    box = offsets * anchors[:, :, None, 3:6]
    s, co = anchors[:, :, None, 6], anchors[:, :, None, 7]
    turned = torch.stack([co * box[..., 0] - s * box[..., 1], s * box[..., 0] + co * box[..., 1], box[..., 2]], -1)
    q = turned + anchors[:, :, None, 0:3] + anchors[:, :, None, 8:11] * dt[:, None, None, None]
    h = [sum(proj[:, None, None, :, r, j] * q[..., None, j] for j in range(3)) + proj[:, None, None, :, r, 3]
         for r in range(3)]
    behind = h[2] <= 1e-5
    z = torch.where(behind, torch.ones_like(h[2]), h[2])
    uv = torch.stack([h[0] / z / img_wh[:, 0], h[1] / z / img_wh[:, 1]], -1)
    return torch.where(behind[..., None], torch.full_like(uv, -2.0), uv)


def _scene_inputs(c, seed, dev):
    gen = torch.Generator(device=dev).manual_seed(seed)
    B, K, A, P, C, G = c["B"], c["cams"], c["A"], c["P"], c["C"], c["G"]
    shape, start, rows = inputs.tables(_cam_maps(c))
    S = shape.shape[1]
    d = dict(case=c, shape=shape.to(dev), start=start.to(dev))
    d["feat"] = torch.empty(B, rows, C, device=dev, dtype=_DT[c["feat"]])
    for b in range(B):
        d["feat"][b] = torch.randn(rows, C, generator=gen, device=dev).mul_(0.5)
    if c["loc"] == "projected":
        d["geometry"] = [t.to(dev) for t in inputs.make_scene_geometry(seed, B, A, P, K)]
        d["loc"] = _project(*d["geometry"]).contiguous()
        away = (d["loc"] < 0).any(-1).any(2) | (d["loc"] > 1).any(-1).any(2)
    else:
        m = c["margin"]
        d["loc"] = torch.rand(B, A, P, K, 2, generator=gen, device=dev) * (1 + 2 * m) - m
        away = torch.rand(B, A, K, generator=gen, device=dev) < c["away"]
        d["loc"][..., 0] += 2.0 * away[:, :, None, :]
    logits = torch.randn(B, A, P * K * S, G, generator=gen, device=dev)
    d["w"] = torch.softmax(logits, dim=2).reshape(B, A, P, K, S, G).to(_DT[c["w"]]).contiguous()
    d["go"] = torch.randn(B, A, C, generator=gen, device=dev)
    if c["kind"] == "oae":
        vis = torch.rand(B, A, K, generator=gen, device=dev)
        d["vis"] = torch.where(away | (torch.rand(B, A, K, generator=gen, device=dev) < 0.1), 0.0, vis).contiguous()
    return d


class _Scene:
    """The tensors of one scene as msda.plan_batched takes them."""

    def __init__(self, d):
        self.feat, self.spatial_shape, self.scale_start_index = d["feat"], d["shape"], d["start"]
        self.sampling_location, self.weights = d["loc"], d["w"]


def prepare(case, seed):
    dev = torch.device("cuda")
    if case["kind"] == "batched":
        scenes = [_scene_inputs(c, seed * 64 + i, dev) for i, c in enumerate(_scenes(case))]
        return dict(case=case, scenes=scenes, plan=msda.plan_batched([_Scene(d) for d in scenes]))
    d = _scene_inputs(case, seed, dev)
    if case["kind"] == "train":
        for n in ("feat", "loc", "w"):
            d[n].requires_grad_()
    if case["kind"] in ("step", "atomic"):  # what a training loop allocates once
        B, rows, C = d["feat"].shape
        _, A, P, K, S, G = d["w"].shape
        need = msda.backward_workspace_size(B, rows, C, K, S, A, P, G, case["kind"] == "step")
        d["out"] = torch.empty(B, A, C, device=dev)
        d["grads"] = (torch.empty(B, rows, C, device=dev), torch.empty(B, A, P, K, 2, device=dev),
                      torch.empty(B, A, P, K, S, G, device=dev))
        d["ws"] = torch.empty(need, dtype=torch.uint8, device=dev)
    return d


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(state):
    d, kind = state, state["case"]["kind"]
    if kind == "batched":
        return d["plan"].run()
    if kind == "serve":
        loc = msda.keypoints(*d["geometry"])
        return [loc, msda.forward(d["feat"], d["shape"], d["start"], loc, d["w"])]
    args = (d["feat"], d["shape"], d["start"], d["loc"], d["w"])
    if kind == "forward":
        return msda.forward(*args)
    if kind == "oae":
        return msda.forward_oae(*args, d["vis"])
    if kind == "train":
        out = msda.msda(*args)
        return [out.detach(), *torch.autograd.grad(out, (d["feat"], d["loc"], d["w"]), d["go"])]
    if kind == "step":
        msda.forward(*args, out=d["out"])
        msda.backward(*args, d["go"], deterministic=True, workspace=d["ws"], grads=d["grads"])
    else:
        msda.forward_train(*args, d["grads"][0], out=d["out"])
        msda.backward(*args, d["go"], workspace=d["ws"], grads=d["grads"], grad_feat_zeroed=True)
    return [d["out"], *d["grads"]]


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def _in_view(c):
    """Share of the point-scales whose bilinear footprint meets its map."""
    if c["loc"] == "projected":
        uv = _project(*inputs.make_scene_geometry(0, 1, 64, min(c["P"], 7), c["cams"]))
        return float(((uv > 0) & (uv < 1)).all(-1).float().mean())
    return (1 - c["away"]) / (1 + 2 * c["margin"]) ** 2


def work(case):
    nbytes = flops = 0.0
    for c in _scenes(case):
        rows = c["B"] * sum(h * w for m in _cam_maps(c) for h, w in m)
        points, anchors = c["B"] * c["A"] * c["P"] * c["cams"], c["B"] * c["A"]
        samples = points * c["scales"] * _in_view(c)
        fsz, wsz = _DT[c["feat"]].itemsize, _DT[c["w"]].itemsize
        once = min(rows, 4 * samples) * c["C"] * fsz + 8 * points + samples * c["G"] * wsz + 4 * anchors * c["C"]
        nbytes += once
        flops += 8 * samples * c["C"]
        if c["kind"] == "serve":
            nbytes += 4 * (11 * anchors + 3 * anchors * c["P"]) + 8 * points
            flops += 40 * points
        if c["kind"] == "oae":
            nbytes += 4 * anchors * c["cams"]
        if c["kind"] in ("train", "step", "atomic"):
            # the backward: the forward's inputs and grad_out again, and the three gradients
            gf, gw = (fsz, wsz) if c["kind"] == "train" else (4, 4)
            nbytes += once + rows * c["C"] * gf + 8 * points + points * c["scales"] * c["G"] * gw
            flops += 16 * samples * c["C"]
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# The same outputs in 64 bits
# ---------------------------------------------------------------------------
def _exact_scene(d, grads=False, loc=None, w=None):
    """out (and the gradients of feat, loc and w) in 64 bits, a map at a time."""
    feat, go = d["feat"].detach(), d["go"].double()
    loc = (d["loc"].detach() if loc is None else loc).double()
    w = (d["w"].detach() if w is None else w).double()
    B, A, P, K, S, G = w.shape
    C = feat.shape[2]
    shape, start = d["shape"].tolist(), d["start"].tolist()
    out = torch.zeros(B, A, C, dtype=torch.float64, device=feat.device)
    if grads:
        gf = torch.zeros(feat.shape, dtype=torch.float64, device=feat.device)
        gl, gw = torch.zeros_like(loc), torch.zeros_like(w)
    for b in range(B):
        for k in range(K):
            for s in range(S):
                H, W = shape[k][s]
                x, y = loc[b, :, :, k, 0] * W - 0.5, loc[b, :, :, k, 1] * H - 0.5
                a, p = ((x > -1) & (x < W) & (y > -1) & (y < H)).nonzero(as_tuple=True)
                x, y = x[a, p], y[a, p]
                x0, y0 = x.floor(), y.floor()
                fx, fy = x - x0, y - y0
                x0, y0 = x0.long(), y0.long()
                wk = w[b, a, p, k, s]  # [N, G]
                wide = wk[:, :, None].expand(-1, G, C // G).reshape(-1, C)
                value, dots = 0.0, []
                gow = go[b, a]
                for j, i, om in ((0, 0, (1 - fx) * (1 - fy)), (1, 0, fx * (1 - fy)), (0, 1, (1 - fx) * fy),
                                 (1, 1, fx * fy)):
                    xi, yi = x0 + j, y0 + i
                    inside = (xi >= 0) & (xi < W) & (yi >= 0) & (yi < H)
                    row = torch.where(inside, start[k][s] + yi * W + xi, 0)
                    F = feat[b, row].double() * inside[:, None]
                    value = value + om[:, None] * F
                    if grads:
                        dots.append((F * gow).reshape(-1, G, C // G).sum(-1))
                        gf[b].index_add_(0, row, wide * gow * (om * inside)[:, None])
                out[b].index_add_(0, a, wide * value)
                if grads:
                    d00, d01, d10, d11 = dots
                    fx, fy = fx[:, None], fy[:, None]
                    gw[b, a, p, k, s] = ((1 - fy) * ((1 - fx) * d00 + fx * d01) + fy * ((1 - fx) * d10 + fx * d11))
                    gl[b, a, p, k, 0] += W * (wk * ((1 - fy) * (d01 - d00) + fy * (d11 - d10))).sum(-1)
                    gl[b, a, p, k, 1] += H * (wk * ((1 - fx) * (d10 - d00) + fx * (d11 - d01))).sum(-1)
    return [out, gf, gl, gw] if grads else out


def exact(case, seed):
    dev = torch.device("cuda")
    if case["kind"] == "batched":
        return [_exact_scene(_scene_inputs(c, seed * 64 + i, dev))[0] for i, c in enumerate(_scenes(case))]
    d = _scene_inputs(case, seed, dev)
    if case["kind"] == "serve":
        loc = _project(*(t.double() for t in d["geometry"]))
        return [loc, _exact_scene(d, loc=loc)]
    if case["kind"] == "oae":
        v = d["vis"].double()
        total = v.sum(-1, keepdim=True)
        share = torch.where(total > 0, v / torch.where(total > 0, total, 1.0), 0.0)
        return _exact_scene(d, w=d["w"].double() * share[:, :, None, :, None, None])
    return _exact_scene(d, grads=case["kind"] in ("train", "step", "atomic"))
