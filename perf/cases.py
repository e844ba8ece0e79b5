"""The calls that are timed when the framework's speed is measured, and what
they compute in 64 bits.

A case is one pass of a user's program through the public entry points:
rendering a frame, a differentiable render, a batch of views, one training
iteration up to its gradients, the full deformation module, the decoder with
its loss, the optimiser.  Scenes follow the distributions of the package's
synthetic generator (uniform means in a box, log-scales N(-3, 0.5), SH
N(0, 0.3), features N(0, 1), planes N(1, 0.1)), drawn on the GPU from the
seed alone.

    listed()             the fixed cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  inputs on the GPU and the objects a program keeps
    run(state)           one pass; its outputs
    work(case)           bytes and operations the pass cannot do without
    exact(case, seed)    the outputs in 64-bit torch (None where too long)
"""
from __future__ import annotations

import math

import torch

from paper_2503_06161_gb300 import _lib
from paper_2503_06161_gb300.batch import BatchRenderer, View
from paper_2503_06161_gb300.decoder import Decoder
from paper_2503_06161_gb300.fst import FSTDeform
from paper_2503_06161_gb300.optim import Adam
from paper_2503_06161_gb300.raster import DeformField, GaussianScene, Rasterizer, render
from paper_2503_06161_gb300.train import LAMBDA_TV, Trainer

DEV = "cuda"
HIDDEN, HEADS, GRID = 64, 11, 64  # single-level deformation field: MLP width, offsets, plane nodes
# Scene boxes: the endoscopic field of the training workloads, and a small
# cube close to the camera.
BOXES = {"field": ((-2.0, -2.0, 3.0), (2.0, 2.0, 8.0)), "near": ((-1.0, -1.0, 2.0), (1.0, 1.0, 4.0))}


def listed():
    return [
        # A preview of a small static scene: the smallest call, where launches
        # and latency count.
        dict(name="view_1k_64x64", kind="view", P=1000, D=16, W=64, H=64, f=80.0, box="near", C=0, bf16=False, t=0.0),
        # Playback of a deforming scene from its bf16 storage, at an odd
        # window size, while the scene is still sparse.
        dict(name="view_30k_333x251_bf16", kind="view", P=30011, D=16, W=333, H=251, f=290.0, box="field", C=32,
             bf16=True, t=0.3),
        # Playback of a deforming scene at the paper's frame size (frames/s).
        dict(name="view_200k_640x512", kind="view", P=200000, D=32, W=640, H=512, f=560.0, box="field", C=32,
             bf16=False, t=0.5),
        # Differentiable render of a toy scene, as in gradient checks and
        # small fits.
        dict(name="grad_1k5_96x72", kind="grad", P=1500, D=32, W=96, H=72, f=84.0, box="field", C=32, t=0.5),
        # The default training render, forward and reverse.
        dict(name="grad_200k_640x512", kind="grad", P=200000, D=32, W=640, H=512, f=560.0, box="field", C=32, t=0.5),
        # The same frame at the paper's 128-wide features and its initial
        # number of points.
        dict(name="grad_90k_640x512_d128", kind="grad", P=90000, D=128, W=640, H=512, f=560.0, box="field", C=32,
             t=0.7),
        # A multi-view training batch at two resolutions, replayed as one graph.
        dict(name="batch_100k_8views", kind="batch", P=100000, D=32, W=640, H=512, f=560.0, box="field", C=32, views=8),
        # One training iteration of a large scene at the native camera
        # resolution: render, losses, decoder, reverse (up to the gradients).
        dict(name="train_1m_1280x1024", kind="train", P=1000000, D=64, W=1280, H=1024, f=1000.0, box="field", C=32,
             t=0.5),
        # The full deformation module at inference.
        dict(name="fst_200k", kind="fst", P=200000, D=32, levels=4, rs=64, rt=100, bf16=False, t=0.4, grad=False),
        # The full deformation module in training: forward, reverse, and the
        # total-variation term.
        dict(name="fst_grad_200k", kind="fst", P=200000, D=32, levels=4, rs=64, rt=100, bf16=True, t=0.4, grad=True),
        # The semantic decoder with the feature loss and its reverse.
        dict(name="decoder_640x512", kind="decoder", HW=640 * 512, D=32, bf16=True),
        # The optimiser over every parameter of the default scene.
        dict(name="adam_200k", kind="adam", P=200000, D=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("view", "view", "grad", "grad", "grad", "batch", "train", "fst", "fst", "fst", "decoder", "adam"))
    W = _log(rng, 64, 1280)
    H = max(48, int(W * rng.uniform(0.7, 0.9)))
    f = round(W * rng.uniform(0.78, 1.25), 2)
    t = round(rng.random(), 3)
    box = "near" if W < 160 else "field"
    if kind == "view":
        return dict(kind=kind, P=_log(rng, 1000, 400000), D=rng.choice((16, 32, 64, 128, 256)), W=W, H=H, f=f, box=box,
                    C=rng.choice((0, 32, 32, 64)), bf16=rng.random() < 0.5, t=t)
    if kind == "grad":
        D = rng.choice((16, 32, 64, 128, 256))
        # The widest features on frames of at most the paper's size.
        W, H, f = (W, H, f) if D <= 64 or W <= 640 else (W // 2, H // 2, f / 2)
        return dict(kind=kind, P=_log(rng, 1000, 300000 if D <= 64 else 120000), D=D, W=W, H=H, f=f, box=box,
                    C=rng.choice((0, 32, 32, 64)), t=t)
    if kind == "batch":
        W = _log(rng, 96, 640)
        return dict(kind=kind, P=_log(rng, 2000, 150000), D=rng.choice((16, 32, 64)), W=W, H=max(64, int(0.8 * W)),
                    f=round(0.875 * W, 2), box="field", C=32, views=rng.randint(2, 8))
    if kind == "train":
        return dict(kind=kind, P=_log(rng, 5000, 700000), D=rng.choice((16, 32, 64)), W=W, H=H, f=f, box=box, C=32, t=t)
    if kind == "fst":
        return dict(kind=kind, P=_log(rng, 1000, 250000), D=rng.choice((16, 32, 64, 128)), levels=rng.randint(1, 4),
                    rs=64, rt=100, bf16=rng.random() < 0.5, t=t, grad=rng.random() < 0.6)
    if kind == "decoder":
        return dict(kind=kind, HW=W * H, D=rng.choice((16, 32, 64, 128)), bf16=rng.random() < 0.7)
    return dict(kind="adam", P=_log(rng, 1000, 1000000), D=rng.choice((16, 32, 64, 128)))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
class _Draws:
    """Seeded draws on the GPU."""

    def __init__(self, seed, salt=0):
        self.g = torch.Generator(device=DEV).manual_seed(1000003 * int(seed) + salt)

    def normal(self, *shape, mean=0.0, std=1.0):
        return torch.randn(*shape, generator=self.g, device=DEV).mul_(std).add_(mean)

    def uniform(self, *shape):
        return torch.rand(*shape, generator=self.g, device=DEV)

    def sign(self, *shape):
        return torch.randint(0, 2, shape, generator=self.g, device=DEV).float().mul_(2.0).sub_(1.0)


def _scene_inputs(c, seed):
    d = _Draws(seed, 1)
    lo, hi = (torch.tensor(v, device=DEV) for v in BOXES[c["box"]])
    P, D = c["P"], c["D"]
    q = d.normal(P, 4)
    return dict(means=lo + (hi - lo) * d.uniform(P, 3), log_scales=d.normal(P, 3, mean=-3.0, std=0.5),
                quats=q / q.norm(dim=1, keepdim=True), opacity_logits=d.normal(P), sh=d.normal(P, 16, 3, std=0.3),
                feat=d.normal(P, D))


def _field_inputs(c, seed):
    """Single-level HexPlane field (None for a static scene)."""
    C = c["C"]
    if not C:
        return None
    d = _Draws(seed, 2)
    wh = d.normal(HEADS, HIDDEN, std=0.01 / 8.0)
    wh[0:3] = 0.0
    wh[10] = 0.0
    z = lambda n: torch.zeros(n, device=DEV)
    return dict(planes=d.normal(6, GRID, GRID, C, mean=1.0, std=0.1), w1=d.normal(HIDDEN, C, std=math.sqrt(2.0 / C)),
                b1=z(HIDDEN), w2=d.normal(HIDDEN, HIDDEN, std=math.sqrt(2.0 / HIDDEN)), b2=z(HIDDEN), wh=wh,
                bh=z(HEADS), noise=d.normal(c["P"], 3), noise_scale=0.01)


def _camera(c, W=None, H=None, f=None):
    W, H, f = W or c["W"], H or c["H"], f or c["f"]
    eye = [1.0, 0, 0, 0, 0, 1.0, 0, 0, 0, 0, 1.0, 0, 0, 0, 0, 1.0]
    return _lib.make_camera(W, H, f, f, W / 2.0, H / 2.0, eye, [0.0, 0.0, 0.0])


def _scene(x, bf16=False):
    st = torch.bfloat16 if bf16 else torch.float32
    return GaussianScene(x["means"], x["log_scales"], x["quats"], x["opacity_logits"], x["sh"].to(st),
                         x["feat"].to(st), 3)


def _field(x, box):
    if x is None:
        return None
    return DeformField(x["planes"], x["w1"], x["b1"], x["w2"], x["b2"], x["wh"], x["bh"], *BOXES[box], x["noise"],
                       x["noise_scale"])


def _upstream(c, seed):
    """Gradients of L1 losses: signs over the pixel count (depth weighted 0.01)."""
    d, HW = _Draws(seed, 3), c["W"] * c["H"]
    return dict(rgb=d.sign(3, c["H"], c["W"]) / HW, depth=d.sign(c["H"], c["W"]) * (0.01 / HW),
                feat=d.sign(HW, c["D"]) / HW)


FST_DEPTH, FST_C, FST_BRANCH = 8, 32, (3, 4, 3, 1)
FST_PAIRS = ((0, 1), (0, 2), (1, 2), (0, 3), (1, 3), (2, 3))


def _fst_layers(levels, D):
    out = [(64, levels * FST_C)] + [(64, 64)] * (FST_DEPTH - 1)
    for d in FST_BRANCH:
        out += [(32, 64), (32, 32), (d, 32)]
    return out + [(64, 128), (D, 64)]


def _fst_planes(levels, rs, rt):
    return [((rs << lv) if a < 3 else rt, (rs << lv) if b < 3 else rt) for lv in range(levels) for a, b in FST_PAIRS]


def _fst_inputs(c, seed):
    d = _Draws(seed, 4)
    shapes = _fst_layers(c["levels"], c["D"])
    parts = []
    for k, (o, i) in enumerate(shapes):
        std = math.sqrt(2.0 / i)
        if k in (10, 13, 16, 19):
            std = 0.01 / math.sqrt(i)
        if k == len(shapes) - 1:
            std = 0.1 / math.sqrt(i)
        parts += [d.normal(o * i, std=std), d.normal(o, std=0.01)]
    n = sum(a * b * FST_C for a, b in _fst_planes(c["levels"], c["rs"], c["rt"]))
    return dict(planes=d.normal(n, mean=1.0, std=0.1), mlp=torch.cat(parts))


def _fst_upstream(c, seed):
    """Gradients of the deformed Gaussians, of the sizes a render's reverse gives."""
    d, P = _Draws(seed, 5), c["P"]
    return dict(means=d.normal(P, 3, std=1e-5), quats=d.normal(P, 4, std=1e-6), log_scales=d.normal(P, 3, std=1e-6),
                opacity_logits=d.normal(P, std=1e-6), feat=d.normal(P, c["D"], std=1e-6))


def _decoder_inputs(c, seed):
    d, D = _Draws(seed, 6), c["D"]
    return dict(feat=d.normal(c["HW"], D).to(torch.bfloat16), weight=d.normal(256, D, std=0.05).to(torch.bfloat16),
                bias=d.normal(256, std=0.05),
                target=d.normal(c["HW"], 256).to(torch.bfloat16 if c["bf16"] else torch.float32))


ADAM_LR = dict(means=1.6e-4, log_scales=5e-3, quats=1e-3, opacity_logits=5e-2, sh=2.5e-3, feat=2.5e-3)


def _adam_inputs(c, seed):
    x = _scene_inputs(dict(c, box="field"), seed)
    d = _Draws(seed, 7)
    g = [{k: d.normal(*x[k].shape, std=1e-6) for k in ADAM_LR} for _ in range(2)]
    return x, g


def _targets(c, seed):
    d = _Draws(seed, 8)
    lo, hi = BOXES[c["box"]]
    rgb = d.uniform(3, c["H"], c["W"])
    dec = d.normal(c["W"] * c["H"], 256).to(torch.bfloat16)
    depth = lo[2] + (hi[2] - lo[2]) * d.uniform(c["H"], c["W"])
    return rgb, dec, depth


# ---------------------------------------------------------------------------
# prepare / run
# ---------------------------------------------------------------------------
def prepare(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind == "view":
        x = _scene_inputs(c, seed)
        return dict(kind=kind, scene=_scene(x, c["bf16"]), field=_field(_field_inputs(c, seed), c["box"]),
                    cam=_camera(c), t=c["t"], rast=Rasterizer(c["P"], c["D"], c["W"], c["H"], forward_only=True))
    if kind == "grad":
        scene = _scene(_scene_inputs(c, seed))
        for p in scene.params():
            p.requires_grad_(True)
        return dict(kind=kind, scene=scene, field=_field(_field_inputs(c, seed), c["box"]), cam=_camera(c), t=c["t"],
                    g=_upstream(c, seed), rast=Rasterizer(c["P"], c["D"], c["W"], c["H"]))
    if kind == "batch":
        views, V = [], c["views"]
        d = _Draws(seed, 9)
        for k in range(V):
            half = k >= (V + 1) // 2
            W, H, f = (c["W"] // 2, c["H"] // 2, c["f"] / 2) if half else (c["W"], c["H"], c["f"])
            views.append(View(_camera(c, W, H, f), k / (V - 1), d.uniform(3, H, W), d.normal(H * W, c["D"])))
        br = BatchRenderer(_scene(_scene_inputs(c, seed), True), _field(_field_inputs(c, seed), c["box"]), views, None)
        br.capture()
        return dict(kind=kind, br=br)
    if kind == "train":
        w = _decoder_inputs(dict(HW=1, D=c["D"], bf16=True), seed)
        tr = Trainer(_scene_inputs(c, seed), 3, _camera(c), _field(_field_inputs(c, seed), c["box"]),
                     Decoder(w["weight"], w["bias"]))
        return dict(kind=kind, tr=tr, t=c["t"], targets=_targets(c, seed))
    if kind == "fst":
        x = _scene_inputs(dict(c, box="field"), seed)
        p = _fst_inputs(c, seed)
        fst = FSTDeform(p["planes"], p["mlp"], c["levels"], c["rs"], c["rt"], c["D"], *BOXES["field"], c["P"],
                        with_backward=c["grad"])
        s = dict(kind=kind, fst=fst, scene=_scene(x, c["bf16"]), t=c["t"], grad=c["grad"])
        if c["grad"]:
            s["up"] = _fst_upstream(c, seed)
            s["g"] = {k: v.clone() for k, v in s["up"].items()}
            s["loss"], s["scratch"] = torch.zeros(1, device=DEV), torch.empty(1024, device=DEV)
        return s
    if kind == "decoder":
        x = _decoder_inputs(c, seed)
        return dict(kind=kind, dec=Decoder(x["weight"], x["bias"]), feat=x["feat"], target=x["target"])
    x, grads = _adam_inputs(c, seed)
    opt = Adam([dict(param=x[k], lr=ADAM_LR[k]) for k in ADAM_LR])
    opt.step([grads[0][k] for k in ADAM_LR])  # moments as in the middle of training
    return dict(kind=kind, opt=opt, grads=[grads[1][k] for k in ADAM_LR])


def run(state):
    kind = state["kind"]
    if kind == "view":
        return state["rast"].forward(state["scene"], state["cam"], state["field"], state["t"])
    if kind == "grad":
        g = state["g"]
        rgb, depth, alpha, feat = render(state["rast"], state["scene"], state["cam"], state["field"], state["t"])
        grads = torch.autograd.grad((rgb, depth, feat), state["scene"].params(), (g["rgb"], g["depth"], g["feat"]))
        return (rgb.detach(), depth.detach(), alpha.detach(), feat.detach()) + tuple(grads)
    if kind == "batch":
        br = state["br"]
        br.replay()
        return dict(grads=br.grads, losses=br.losses, images=[b["out"] for b in br.bufs])
    if kind == "train":
        tr = state["tr"]
        tr.forward_backward(state["t"], *state["targets"])
        return dict(losses=tr.losses, images=tr.out, feat_bf16=tr.feat_bf, grads=tr.grads, decoder=tr.dec_out[1:])
    if kind == "fst":
        fst, scene, t = state["fst"], state["scene"], state["t"]
        o = fst.forward(scene, t)
        out = dict(means=o.means, quats=o.quats, log_scales=o.log_scales, opacity_logits=o.opacity_logits, feat=o.feat)
        if state["grad"]:
            state["g"]["means"].copy_(state["up"]["means"])  # the render's reverse rewrites it every iteration
            fst.backward(scene, t, state["g"])
            fst.tv(LAMBDA_TV, state["loss"], state["scratch"])
            out.update(d_means=state["g"]["means"], d_planes=fst.d_planes, d_mlp=fst.d_mlp, tv=state["loss"])
        return out
    if kind == "decoder":
        return state["dec"].l1(state["feat"], state["target"])
    opt = state["opt"]
    opt.step(state["grads"])
    return [[g["param"], g["m"], g["v"]] for g in opt.groups]


# ---------------------------------------------------------------------------
# Work
# ---------------------------------------------------------------------------
def _blended(P, HW, f):
    """Gaussians blended per pixel: the expected cover of the box's
    footprints, up to the about 72 that make a pixel of a dense scene opaque
    (measured on the 200k-Gaussian frame)."""
    return min(72.0, 72.0 * P * f * f / (30000 * 560.0 ** 2) * (640 * 512) / HW)


def _view_work(c, W, H, f, backward, bf16):
    P, D, C, HW = c["P"], c["D"], c["C"], W * H
    e = 2 if bf16 else 4
    pairs = _blended(P, HW, f) * HW
    by = P * (11 * 4 + 48 * e + D * e) + HW * (5 + D) * 4
    fl = 450.0 * P + pairs * (18 + 2 * (4 + D))
    if C:
        by += 6 * GRID * GRID * C * 4 + P * 12
        fl += P * (2.0 * (HIDDEN * C + HIDDEN * HIDDEN + HEADS * HIDDEN) + 54 * C)
    if backward:
        by += HW * (4 + D) * 4 + P * (11 + 48 + D) * 4
        fl += 1050.0 * P + pairs * (14 + 2 * (4 + D) + 35 + 2 * (10 + D))
        if C:
            fl += P * (2.0 * (HIDDEN * C + HIDDEN * HIDDEN + HEADS * HIDDEN) + 198 * C)
    return by, fl


def work(case):
    c = case
    kind = c["kind"]
    if kind in ("view", "grad"):
        by, fl = _view_work(c, c["W"], c["H"], c["f"], kind == "grad", c.get("bf16", False))
    elif kind == "batch":
        by = fl = 0.0
        for k in range(c["views"]):
            s = 2 if k >= (c["views"] + 1) // 2 else 1
            b, n = _view_work(c, c["W"] // s, c["H"] // s, c["f"] / s, True, True)
            by, fl = by + b - c["P"] * (11 + 48 + c["D"]) * 4 * (k > 0), fl + n  # one summed set of gradients
    elif kind == "train":
        HW = c["W"] * c["H"]
        by, fl = _view_work(c, c["W"], c["H"], c["f"], True, True)
        by += HW * (256 * 2 + 4 * 4)
        fl += HW * 6.0 * 256 * c["D"]
    elif kind == "fst":
        P, D, L = c["P"], c["D"], c["levels"]
        n = sum(a * b * FST_C for a, b in _fst_planes(L, c["rs"], c["rt"]))
        macs = sum(o * i for o, i in _fst_layers(L, D))
        by = P * 2 * (11 * 4 + D * (2 if c["bf16"] else 4)) + 4 * (n + macs)
        fl = P * (2.0 * macs + 54 * FST_C * L)
        if c["grad"]:
            by += P * (14 + D) * 4 + 4 * (n + macs)
            fl += P * (4.0 * macs + 198 * FST_C * L) + 12 * n
    elif kind == "decoder":
        by = c["HW"] * (c["D"] * 2 + 256 * (2 if c["bf16"] else 4) + c["D"] * 4) + 256 * (6 * c["D"] + 8)
        fl = c["HW"] * 6.0 * 256 * c["D"]
    else:
        n = c["P"] * (11 + 48 + c["D"])
        by, fl = 28 * n, 12 * n
    return {"bytes": float(by), "flops": float(fl)}


# ---------------------------------------------------------------------------
# 64-bit values
# ---------------------------------------------------------------------------
def _bilinear(plane, x, y):
    """Bilinear samples of a channels-last plane at node positions x, y >= 0."""
    i = x.detach().floor().long().clamp_(0, plane.shape[0] - 2)
    j = y.detach().floor().long().clamp_(0, plane.shape[1] - 2)
    fx, fy = (x - i)[:, None], (y - j)[:, None]
    return (1 - fx) * ((1 - fy) * plane[i, j] + fy * plane[i, j + 1]) + \
        fx * ((1 - fy) * plane[i + 1, j] + fy * plane[i + 1, j + 1])


def _node(mu, lo, hi, R):
    """Positions on R nodes spanning [lo, hi], clamped to the border."""
    return ((mu - lo) / (hi - lo) * (R - 1)).clamp(0, R - 1)


def _offsets64(field, box, mu, t):
    lo, hi = BOXES[box]
    w = {k: v.double() for k, v in field.items() if torch.is_tensor(v)}
    pos = [_node(mu[:, k], lo[k], hi[k], GRID) for k in range(3)]
    pos.append(torch.full_like(pos[0], min(max(t, 0.0), 1.0) * (GRID - 1)))
    f = 1.0
    for k, (a, b) in enumerate(FST_PAIRS):
        f = f * _bilinear(w["planes"][k], pos[a], pos[b])
    h = torch.relu(f @ w["w1"].T + w["b1"])
    h = torch.relu(h @ w["w2"].T + w["b2"])
    d = h @ w["wh"].T + w["bh"]
    return torch.cat([d[:, :3] + field["noise_scale"] * t * w["noise"], d[:, 3:]], 1)


def _sh64(d):
    """Real spherical harmonics to degree 3 with the Condon-Shortley phase."""
    x, y, z = d.unbind(1)
    pi = math.pi
    k1, k2 = math.sqrt(3 / (4 * pi)), math.sqrt(15 / (4 * pi))
    a3, b3, c3, d3, e3 = (math.sqrt(v / pi) for v in (35 / 32, 105 / 4, 21 / 32, 7 / 16, 105 / 16))
    return torch.stack([
        torch.full_like(x, 0.5 / math.sqrt(pi)), -k1 * y, k1 * z, -k1 * x, k2 * x * y, -k2 * y * z,
        math.sqrt(5 / (16 * pi)) * (2 * z * z - x * x - y * y), -k2 * x * z, 0.5 * k2 * (x * x - y * y),
        -a3 * y * (3 * x * x - y * y), b3 * x * y * z, -c3 * y * (4 * z * z - x * x - y * y),
        d3 * z * (2 * z * z - 3 * x * x - 3 * y * y), -c3 * x * (4 * z * z - x * x - y * y), e3 * z * (x * x - y * y),
        -a3 * x * (x * x - 3 * y * y)], 1)


def _project64(c, p, delta):
    """Screen-space Gaussians of an identity camera: columns u, v, conic a b c,
    opacity, depth, r g b, features; their radii; the order by depth of those
    on screen."""
    W, H, f = c["W"], c["H"], c["f"]
    mu, q, ls, lg = p["means"], p["quats"], p["log_scales"], p["opacity_logits"]
    if delta is not None:
        mu, q, ls, lg = mu + delta[:, :3], q + delta[:, 3:7], ls + delta[:, 7:10], lg + delta[:, 10]
    q = q / q.norm(dim=1, keepdim=True)
    w, x, y, z = q.unbind(1)
    R = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                     2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                     2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    M = R * ls.exp()[:, None, :]
    S = M @ M.transpose(1, 2)
    zc = mu[:, 2]
    tx, ty = mu[:, 0] / zc, mu[:, 1] / zc
    lx, ly = 1.3 * 0.5 * W / f, 1.3 * 0.5 * H / f
    zero = torch.zeros_like(zc)
    T = torch.stack([f / zc, zero, -f * tx.clamp(-lx, lx) / zc, zero, f / zc, -f * ty.clamp(-ly, ly) / zc], 1)
    T = T.view(-1, 2, 3)
    cov = T @ S @ T.transpose(1, 2)
    a, b, cc = cov[:, 0, 0] + 0.3, cov[:, 0, 1], cov[:, 1, 1] + 0.3
    det = a * cc - b * b
    mid = 0.5 * (a + cc)
    radius = torch.ceil(3 * torch.sqrt(mid + torch.sqrt((mid * mid - det).clamp_min(0.1)))).detach()
    u, v = f * tx + W / 2.0, f * ty + H / 2.0
    rgb = (torch.einsum("pk,pkc->pc", _sh64(mu / mu.norm(dim=1, keepdim=True)), p["sh"]) + 0.5).clamp_min(0.0)
    rec = torch.cat([torch.stack([u, v, cc / det, -b / det, a / det, torch.sigmoid(lg), zc], 1), rgb, p["feat"]], 1)
    seen = (zc > 0.2) & (u + radius > 0) & (u - radius < W) & (v + radius > 0) & (v - radius < H)
    ids = torch.nonzero(seen.detach())[:, 0]
    # Depths are compared as the 32-bit values that order the pass.
    return rec, radius, ids[torch.sort(zc.detach()[ids].float(), stable=True).indices]


def _tile64(r, radius, px, py):
    """(rgb, depth, alpha, features) at pixel centres px, py of depth-ordered records."""
    dx, dy = px[:, None] - r[None, :, 0], py[:, None] - r[None, :, 1]
    power = -0.5 * (r[:, 2] * dx * dx + r[:, 4] * dy * dy) - r[:, 3] * dx * dy
    G = torch.exp(power.clamp_max(0.0))
    al = r[:, 5] * G
    over = al > 0.99  # a clamped alpha keeps its opacity gradient
    flat = r[:, 5] * G.detach()
    al = torch.where(over, 0.99 + flat - flat.detach(), al)
    keep = (dx.abs() <= radius) & (dy.abs() <= radius) & (power <= 0) & (al >= 1.0 / 255.0)
    al = torch.where(keep.detach(), al, torch.zeros_like(al))
    live = torch.cumprod(1 - al.detach(), 1) >= 1e-4
    al = al * live
    T = torch.cumprod(1 - al, 1)
    w = al * torch.cat([torch.ones_like(T[:, :1]), T[:, :-1]], 1)
    out = w @ r[:, 6:]
    return out[:, 1:4], out[:, 0], 1 - T[:, -1], out[:, 4:]


def _render64(c, scene, field, up):
    W, H, D = c["W"], c["H"], c["D"]
    names = ("means", "log_scales", "quats", "opacity_logits", "sh", "feat")
    st = torch.bfloat16 if c.get("bf16") else torch.float32
    p = {k: (scene[k].to(st) if k in ("sh", "feat") else scene[k]).double() for k in names}
    if up is not None:
        p = {k: v.requires_grad_(True) for k, v in p.items()}
    with torch.set_grad_enabled(up is not None):
        delta = _offsets64(field, c["box"], p["means"], c["t"]) if field is not None else None
        rec, radius, order = _project64(c, p, delta)
    base = rec.detach()
    k64 = dict(dtype=torch.float64, device=DEV)
    rgb, depth, alpha = torch.zeros(3, H, W, **k64), torch.zeros(H, W, **k64), torch.zeros(H, W, **k64)
    feat, d_rec = torch.zeros(H, W, D, **k64), torch.zeros_like(base)
    ou, ov, orad = base[order, 0], base[order, 1], radius[order]
    for y0 in range(0, H, 16):
        y1 = min(H, y0 + 16)
        row = (ov + orad >= y0 + 0.5) & (ov - orad <= y1 - 0.5)
        for x0 in range(0, W, 16):
            x1 = min(W, x0 + 16)
            ids = order[row & (ou + orad >= x0 + 0.5) & (ou - orad <= x1 - 0.5)]
            if not len(ids):
                continue
            py, px = torch.meshgrid(torch.arange(y0, y1, **k64) + 0.5, torch.arange(x0, x1, **k64) + 0.5, indexing="ij")
            r = base[ids].requires_grad_(up is not None)
            with torch.set_grad_enabled(up is not None):
                o = _tile64(r, radius[ids], px.reshape(-1), py.reshape(-1))
            at, n = (slice(y0, y1), slice(x0, x1)), (y1 - y0, x1 - x0)
            rgb[(slice(None),) + at] = o[0].detach().T.reshape(3, *n)
            depth[at], alpha[at] = o[1].detach().view(n), o[2].detach().view(n)
            feat[at] = o[3].detach().view(*n, D)
            if up is not None:
                g = (up["rgb"][(slice(None),) + at].reshape(3, -1).T.double(), up["depth"][at].reshape(-1).double(),
                     up["feat"].view(H, W, D)[at].reshape(-1, D).double())
                d_rec.index_add_(0, ids, torch.autograd.grad((o[0], o[1], o[3]), r, g)[0])
    out = (rgb, depth, alpha, feat.view(H * W, D))
    if up is None:
        return out
    return out + torch.autograd.grad(rec, [p[k] for k in names], d_rec)


def _fst64(c, x, p, up):
    L, rs, rt, D, t = c["levels"], c["rs"], c["rt"], c["D"], c["t"]
    lo, hi = BOXES["field"]
    st = torch.bfloat16 if c["bf16"] else torch.float32
    planes, mlp, mu = (v.double().requires_grad_(c["grad"]) for v in (p["planes"], p["mlp"], x["means"]))
    with torch.set_grad_enabled(c["grad"]):
        fs, off, tv = [], 0, 0.0
        for lv in range(L):
            f = 1.0
            for k, (a, b) in enumerate(FST_PAIRS):
                ra, rb = _fst_planes(L, rs, rt)[lv * 6 + k]
                pl = planes[off:off + ra * rb * FST_C].view(ra, rb, FST_C)
                off += pl.numel()
                pa = _node(mu[:, a], lo[a], hi[a], ra)
                pb = _node(mu[:, b], lo[b], hi[b], rb) if b < 3 else torch.full_like(pa, t * (rt - 1))
                f = f * _bilinear(pl, pa, pb)
                if c["grad"]:
                    tv = tv + (pl[1:] - pl[:-1]).square().mean() + (pl[:, 1:] - pl[:, :-1]).square().mean()
            fs.append(f)
        ws, off = [], 0
        for o, i in _fst_layers(L, D):
            ws.append((mlp[off:off + o * i].view(o, i), mlp[off + o * i:off + o * i + o]))
            off += o * i + o
        lin = lambda k, v: v @ ws[k][0].T + ws[k][1]
        h = lin(0, torch.cat(fs, 1))
        for k in range(1, FST_DEPTH):
            h = lin(k, torch.relu(h))
        us, heads = [], []
        for b in range(4):
            k = FST_DEPTH + 3 * b
            u = lin(k + 1, torch.relu(lin(k, torch.relu(h))))
            us.append(u)
            heads.append(lin(k + 2, torch.relu(u)))
        dz = lin(21, torch.relu(lin(20, torch.relu(torch.cat(us, 1)))))
        out = dict(means=mu + heads[0], quats=x["quats"].double() + heads[1],
                   log_scales=x["log_scales"].double() + heads[2],
                   opacity_logits=x["opacity_logits"].double() + heads[3][:, 0], feat=x["feat"].to(st).double() + dz)
        if c["grad"]:
            names = list(out)
            tv = LAMBDA_TV * tv
            g = torch.autograd.grad([out[k] for k in names] + [tv], [mu, planes, mlp],
                                    [up[k].double() for k in names] + [torch.ones_like(tv)])
            out.update(d_means=g[0], d_planes=g[1], d_mlp=g[2], tv=tv.detach().view(1))
    return {k: v.detach() for k, v in out.items()}


def exact(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind in ("view", "grad"):
        # One pass over the tiles, each against its own list: bounded by the
        # number of tiles and by the length of the lists.
        if c["W"] * c["H"] > 700_000 or c["P"] > 250_000:
            return None
        return _render64(c, _scene_inputs(c, seed), _field_inputs(c, seed), _upstream(c, seed) if kind == "grad" else None)
    if kind == "fst":
        return _fst64(c, _scene_inputs(dict(c, box="field"), seed), _fst_inputs(c, seed), _fst_upstream(c, seed))
    if kind == "decoder":
        x = {k: v.double() for k, v in _decoder_inputs(c, seed).items()}
        s = 1.0 / c["HW"]
        diff = x["feat"] @ x["weight"].T + x["bias"] - x["target"]
        sg = torch.sign(diff) * s
        return (diff.abs().sum() * s).view(1), sg @ x["weight"], sg.T @ x["feat"], sg.sum(0)
    if kind == "adam":
        x, grads = _adam_inputs(c, seed)
        out = []
        for k in ADAM_LR:
            p, m, v = x[k].double(), 0.0, 0.0
            for step in (1, 2):
                g = grads[step - 1][k].double()
                m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
                p = p - ADAM_LR[k] * (m / (1 - 0.9 ** step)) / ((v / (1 - 0.999 ** step)).sqrt() + 1e-15)
            out.append([p, m, v])
        return out
    return None  # batches and training iterations: too many tiles for a short reference
