"""The forward compositing around the tile counts where its default batch
size (D = 32) and its blocks per SM (D = 16) change: images and gradients are
the same bits as with each batch size set by hand, for one view and for a
batch of views."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2503_06161_gb300 import _lib, synth  # noqa: E402
from paper_2503_06161_gb300.batch import BatchRenderer, View  # noqa: E402
from paper_2503_06161_gb300.raster import GaussianScene, Rasterizer, camera_struct  # noqa: E402

from gpu_helpers import GRAD_KEYS  # noqa: E402


def _scene(P, D, bf16):
    sc = synth.make_scene(P, D, (-1.2, -0.8, 2.0), (1.2, 0.8, 4.5), seed=D)
    return GaussianScene.from_numpy(sc, "cuda", bf16=bf16)


# 342 | 345 tiles and 456 | 460, the last columns and rows ragged.
@pytest.mark.parametrize("D,W,H", [(16, 285, 300), (16, 365, 235), (16, 16, 16), (32, 380, 300), (32, 318, 361),
                                   (32, 9, 5)])
@pytest.mark.parametrize("bf16", [False, True])
def test_defaults_change_no_bit(D, W, H, bf16):
    scene = _scene(6000, D, bf16)
    cam = camera_struct(synth.make_camera(W, H, 0.8 * W))
    gen = torch.Generator(device="cuda").manual_seed(1)
    g = [torch.randn(s, generator=gen, device="cuda") for s in ((3, H, W), (H, W), (H, W), (H * W, D))]
    want = None
    for B in (0, 32, 64, 128):
        rast = Rasterizer(scene.P, D, W, H, bg=(0.1, 0.2, 0.3), fwd_batch=B)
        out = list(rast.forward(scene, cam, None, 0.0))
        rast.check()
        grads = rast.backward(scene, cam, None, 0.0, *g)
        out += [grads[k] for k in GRAD_KEYS]
        if want is None:
            want = out
        assert all(torch.equal(a, b) for a, b in zip(out, want)), B
    assert want[3].abs().max() > 0


@pytest.mark.parametrize("D,sizes", [(16, ((285, 300),)), (16, ((285, 300), (48, 16))), (32, ((380, 300),)),
                                     (32, ((380, 300), (64, 16)))])
def test_batch_defaults_change_no_bit(D, sizes):
    scene = _scene(6000, D, True)
    gen = torch.Generator(device="cuda").manual_seed(2)
    views = [View(camera_struct(synth.make_camera(W, H, 0.8 * W)), 0.0,
                  torch.rand(3, H, W, generator=gen, device="cuda"),
                  torch.randn(H * W, D, generator=gen, device="cuda")) for W, H in sizes]
    want = None
    for B in (0, 32, 64, 128):
        br = BatchRenderer(scene, None, views, None, fwd_batch=B)
        br.run()
        torch.cuda.synchronize()
        assert br.device_errors() == 0
        out = [x.clone() for b in br.bufs for x in b["out"]] + [br.grads[k].clone() for k in GRAD_KEYS]
        if want is None:
            want = out
        assert all(torch.equal(a, b) for a, b in zip(out, want)), B
