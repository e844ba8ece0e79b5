"""Gradients through render(): a loss on some of the outputs alone, whose
other upstream gradients reach the reverse as None, gives bit for bit what
explicit zeros give, and the oracle's gradients."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import oracle as O  # noqa: E402
from paper_2503_06161_gb300.raster import Rasterizer, render  # noqa: E402

from gpu_helpers import GRAD_KEYS, check_grads, deformed_case, forward_parity, gpu_forward, grad_parity  # noqa: E402

NAMES = ("rgb", "depth", "alpha", "feat")
BG = (0.2, 0.1, 0.3)


def _upstream(W, H, D):
    gen = torch.Generator(device="cuda").manual_seed(3)
    return {k: torch.randn(s, generator=gen, device="cuda")
            for k, s in dict(rgb=(3, H, W), depth=(H, W), alpha=(H, W), feat=(H * W, D)).items()}


@pytest.mark.parametrize("D", [32, 128, 256])
@pytest.mark.parametrize("used", [("rgb",), ("depth",), ("alpha",), ("feat",), ("rgb", "feat"), NAMES])
def test_unused_outputs_are_zero_upstream(used, D):
    sc, cam, df = deformed_case(P=1500, W=90, H=70, D=D, f=75.0)
    run = gpu_forward(sc, cam, df, 0.4, bg=BG)
    up = _upstream(90, 70, D)
    for p in run.scene.params():
        p.requires_grad_(True)
    out = dict(zip(NAMES, render(run.rast, run.scene, run.cam, run.deform, 0.4)))
    got = torch.autograd.grad([out[k] for k in used], run.scene.params(), [up[k] for k in used])
    zeros = {k: up[k] if k in used else torch.zeros_like(up[k]) for k in NAMES}
    want = run.rast.backward(run.scene, run.cam, run.deform, 0.4, *[zeros[k] for k in NAMES])
    for k, g in zip(GRAD_KEYS, got):
        assert torch.equal(g, want[k]), k
    if used != ("depth",):
        assert got[0].abs().max() > 0
    if "feat" not in used:
        assert not got[5].any()


def test_no_upstream_gradient_gives_zeros():
    sc, cam, df = deformed_case(P=700, W=64, H=48, D=32, f=60.0)
    run = gpu_forward(sc, cam, df, 0.4, bg=BG)
    g = run.rast.backward(run.scene, run.cam, run.deform, 0.4)
    assert all(not g[k].any() for k in GRAD_KEYS)


@pytest.mark.parametrize("D,used", [(32, ("rgb", "feat")), (32, ("alpha",)), (128, ("feat",)), (128, ("depth",))])
def test_gradients_match_oracle(D, used):
    W, H, t = 90, 70, 0.4
    sc, cam, df = deformed_case(P=1500, W=W, H=H, D=D, f=75.0)
    run = gpu_forward(sc, cam, df, t, bg=BG)
    _, _, flip = forward_parity(run, sc, cam, df, t, BG)
    up = _upstream(W, H, D)
    for p in run.scene.params():
        p.requires_grad_(True)
    rast = Rasterizer(sc.P, D, W, H, bg=BG)
    out = dict(zip(NAMES, render(rast, run.scene, run.cam, run.deform, t)))
    loss = sum((out[k] * up[k]).sum() for k in used)
    loss.backward()
    got = {k: p.grad.cpu().numpy() for k, p in zip(GRAD_KEYS, run.scene.params())}
    G = {k: np.zeros(s) for k, s in dict(rgb=(H * W, 3), depth=H * W, alpha=H * W, feat=(H * W, D)).items()}
    for k in used:
        x = up[k].cpu().numpy().astype(np.float64)
        G[k] = x.reshape(3, -1).T if k == "rgb" else x.reshape(G[k].shape)
    errs, rep = grad_parity(got, sc, cam, df, t, BG, O.all_pixels(W, H), G, flip)
    check_grads(errs, rep)
