"""The products with operands of three BF16 terms are as exact as FP32 ones:
each kernel's error against 64 bits, next to what two terms would give on the
same inputs (emulated here in float64, the operands alone rounded).

Two terms leave 2^-17 of an operand, three and FP32 2^-24 or less, so half of
the two-term error is a bar that a lost term fails and that FP32 rounding
(sums of at most a few hundred products, chains of about twenty layers or
forty blends, some 2^-22 in all) stays well under."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import fst as OF  # noqa: E402
from paper_2503_06161_gb300 import _lib, synth  # noqa: E402
from paper_2503_06161_gb300.fst import FSTDeform  # noqa: E402
from paper_2503_06161_gb300.raster import GaussianScene  # noqa: E402

from gpu_helpers import gpu_backward, gpu_forward  # noqa: E402

LO, HI = (-2.0, -2.0, 3.0), (2.0, 2.0, 8.0)
RELU_MARGIN, CELL_MARGIN = 3e-5, 1e-4


def _bf16(x):
    u = np.ascontiguousarray(x, np.float32).view(np.uint32).astype(np.uint64)
    u = (u + 0x7FFF + ((u >> 16) & 1)) & 0xFFFF0000
    return u.astype(np.uint32).view(np.float32).astype(np.float64)


def two(x):
    """x as the sum of two BF16 terms."""
    x = np.asarray(x, np.float64)
    hi = _bf16(x)
    return hi + _bf16(x - hi)


class Two(np.ndarray):
    """An array whose matrix products take two-term operands."""

    def __matmul__(self, other):
        return np.matmul(two(self), two(other)).view(Two)

    def __rmatmul__(self, other):
        return np.matmul(two(other), two(self)).view(Two)


def rms(x):
    return float(np.sqrt(np.mean(np.square(np.asarray(x, np.float64)))))


def _check(what, got, exact, emulated):
    e, e2 = rms(got - exact) / rms(exact), rms(np.asarray(emulated) - exact) / rms(exact)
    print(f"{what}: error {e:.2e}, two terms {e2:.2e}")
    assert e < 0.5 * e2, what


def _fst(P, levels, rs, rt, D, with_backward):
    sc = synth.make_scene(P, D, LO, HI, seed=21)
    planes, mlp = synth.make_fst(levels, rs, rt, D, seed=22, plane_std=0.2, head_std=0.5, dz_std=0.5, bias_std=0.1)
    scene = GaussianScene.from_numpy(sc, "cuda")
    for x in (scene.quats, scene.log_scales, scene.opacity_logits, scene.feat):
        x.zero_()  # the outputs are the offsets
    fst = FSTDeform.from_numpy(planes, mlp, levels, rs, rt, D, LO, HI, P, with_backward=with_backward)
    layers = OF.unpack_mlp(mlp, levels, D)
    return sc, scene, fst, OF.unpack_planes(planes, levels, rs, rt), layers, [(w.view(Two), b) for w, b in layers]


@pytest.mark.parametrize("levels,D", [(4, 32), (1, 128)])
def test_forward_only_module(levels, D):
    P, rs, rt, t = 512, 8, 6, 0.43
    sc, scene, fst, pl, layers, layers2 = _fst(P, levels, rs, rt, D, False)
    o = fst.forward(scene, t)
    torch.cuda.synchronize()
    mu = np.asarray(sc.means, np.float64)
    ref = OF.forward(pl, layers, mu, t, LO, HI, levels, rs, rt)
    emu = OF.forward(pl, layers2, mu, t, LO, HI, levels, rs, rt)
    for k, x in dict(dq=o.quats, ds=o.log_scales, do=o.opacity_logits, dz=o.feat).items():
        _check(k, x.cpu().numpy().astype(np.float64), ref[k], emu[k])


@pytest.mark.parametrize("levels,D", [(4, 32), (1, 128)])
def test_module_reverse(levels, D):
    P, rs, rt, t = 512, 8, 6, 0.43
    sc, scene, fst, pl, layers, layers2 = _fst(P, levels, rs, rt, D, True)
    fst.forward(scene, t)
    st = OF.forward(pl, layers, np.asarray(sc.means, np.float64), t, LO, HI, levels, rs, rt)["state"]
    drop = OF.margins(st)[0] < RELU_MARGIN
    for lv in range(levels):
        x = (st["coord"][:, :3] + 1.0) * 0.5 * ((rs << lv) - 1)
        drop |= np.abs(x - np.round(x)).min(axis=1) < CELL_MARGIN
    rng = np.random.default_rng(23)
    up = dict(means=rng.normal(size=(P, 3)), quats=rng.normal(size=(P, 4)), log_scales=rng.normal(size=(P, 3)),
              opacity_logits=rng.normal(size=P), feat=rng.normal(size=(P, D)))
    up = {k: v.astype(np.float32).astype(np.float64) for k, v in up.items()}
    for k in up:
        up[k][drop] = 0.0
    g = {k: torch.tensor(v, dtype=torch.float32, device="cuda").contiguous() for k, v in up.items()}
    fst.backward(scene, t, g)
    torch.cuda.synchronize()
    args = [up[k] for k in ("means", "quats", "log_scales", "opacity_logits", "feat")]
    ref = OF.backward(pl, layers, st, *args)
    emu = OF.backward(pl, layers2, st, *args)
    got_w, off, e, e2 = fst.d_mlp.cpu().numpy().astype(np.float64), 0, [], []
    for j, ((dw, db), (dw2, _)) in enumerate(zip(ref["layers"], emu["layers"])):
        e.append(rms(got_w[off:off + dw.size].reshape(dw.shape) - dw) / rms(dw))
        e2.append(rms(np.asarray(dw2) - dw) / rms(dw))
        off += dw.size + db.size
    print("weight gradients", [f"{a:.1e}/{b:.1e}" for a, b in zip(e, e2)])
    # (The emulation keeps a few layers' operands exact: those without a
    # two-term error of the expected size are left out.)
    used = [k for k in range(len(e)) if e2[k] > 2.0 ** -20]
    assert len(used) >= len(e) - 6
    assert all(e[k] < 0.5 * e2[k] for k in used)
    cat = lambda x: np.concatenate([np.asarray(p, np.float64).ravel() for p in x])
    _check("planes", fst.d_planes.cpu().numpy().astype(np.float64), cat(ref["planes"]), cat(emu["planes"]))
    # The path through the coordinates alone (upstream added by the kernel).
    d_mu = g["means"].cpu().numpy().astype(np.float64) - up["means"]
    _check("means", d_mu, ref["mu"], np.asarray(emu["mu"]))


@pytest.mark.parametrize("D", [16, 32, 64, 128])
def test_reverse_compositing(D):
    # Faint Gaussians over the whole image: every pixel blends every one, and
    # no decision is near its threshold.  64-bit reference from the forward's
    # own records, so that only the reverse's arithmetic differs.
    P, W, H = 40, 40, 24
    sc = synth.make_scene(P, D, (-0.3, -0.3, 3.0), (0.3, 0.3, 8.0), seed=31)
    sc.log_scales[:] = 1.6 + 0.2 * (sc.log_scales + 3.0)
    sc.opacity_logits[:] = -2.5 + 0.2 * sc.opacity_logits
    cam = synth.make_camera(W, H, 0.9 * W)
    run = gpu_forward(sc, cam)
    d = {k: v.cpu().numpy().astype(np.float64) for k, v in run.rast.dump().items() if torch.is_tensor(v)}
    order = np.argsort(d["depth"], kind="stable")
    y, x = np.divmod(np.arange(W * H), W)
    dx = (x + 0.5)[:, None] - d["uv"][order, 0]
    dy = (y + 0.5)[:, None] - d["uv"][order, 1]
    ca, cb, cc = d["conic"][order].T
    alpha = d["opacity"][order] * np.exp(-0.5 * (ca * dx * dx + cc * dy * dy) - cb * dx * dy)
    assert 2.0 / 255 < alpha.min() and alpha.max() < 0.9
    assert (np.abs(dx) < d["radius"][order] - 1).all() and (np.abs(dy) < d["radius"][order] - 1).all()
    T = np.cumprod(np.concatenate([np.ones((W * H, 1)), 1.0 - alpha], axis=1), axis=1)
    assert T.min() > 1e-3
    Tf, T = T[:, -1:], T[:, :-1]
    w = alpha * T
    rng = np.random.default_rng(32)
    G = {k: rng.normal(size=s).astype(np.float32).astype(np.float64)
         for k, s in dict(rgb=(W * H, 3), depth=W * H, alpha=W * H, feat=(W * H, D)).items()}
    feat = np.asarray(sc.feat, np.float64)[order]

    def reverse(r):
        s = r(G["feat"]) @ r(feat).T + r(G["rgb"]) @ r(d["rgb"][order]).T + np.outer(G["depth"], d["depth"][order])
        ws = w * s
        Q = np.cumsum(ws[:, ::-1], axis=1)[:, ::-1] - ws
        e = r((T * s - (Q - (G["alpha"][:, None] * Tf)) / (1.0 - alpha)) * alpha)
        du, dv = (e * (ca * dx + cb * dy)).sum(0), (e * (cb * dx + cc * dy)).sum(0)
        return r(w).T @ r(G["feat"]), np.hypot(0.5 * W * du, 0.5 * H * dv), e.sum(0) * (1.0 - d["opacity"][order])

    exact, emu = reverse(lambda a: a), reverse(two)
    got = gpu_backward(run, 0.0, G["rgb"], G["depth"], G["alpha"], G["feat"])
    accum, count = torch.zeros(P, device="cuda"), torch.zeros(P, dtype=torch.int32, device="cuda")
    _lib.fe_screen_grad_stats(run.rast.workspace, P, D, W, H, run.rast.opts, accum, count)
    stat = accum.cpu().numpy().astype(np.float64)
    _check("features", got["feat"].astype(np.float64)[order], exact[0], emu[0])
    _check("centres", stat[order], exact[1], emu[1])
    _check("opacities", got["opacity_logits"].astype(np.float64)[order], exact[2], emu[2])
