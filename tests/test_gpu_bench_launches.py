"""The launch counts that bench.py reports against a trace of the same calls."""
import os
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402
from paper_2503_06161_gb300 import synth  # noqa: E402
from paper_2503_06161_gb300.batch import BatchRenderer, View  # noqa: E402
from paper_2503_06161_gb300.decoder import Decoder  # noqa: E402
from paper_2503_06161_gb300.raster import DeformField, GaussianScene, Rasterizer, camera_struct  # noqa: E402


def _launches(fn):
    fn()
    torch.cuda.synchronize()
    for _ in range(3):  # (the first trace of a process may come back empty)
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
            fn()
            torch.cuda.synchronize()
        names = [e.name for e in prof.events() if e.device_type == torch.autograd.DeviceType.CUDA]
        if names:
            break
    if not names:
        pytest.skip("no kernel trace on this machine")
    return sum("fe::" in n for n in names)


def _case(P, D, deform):
    sc = synth.make_scene(P, D, (-1.2, -0.8, 2.0), (1.2, 0.8, 4.5), seed=0)
    df = synth.make_deform(P, C=32, R=16, bbox_min=(-1.5, -1.0, 1.5), bbox_max=(1.5, 1.0, 5.0)) if deform else None
    return GaussianScene.from_numpy(sc, "cuda", bf16=True), DeformField.from_numpy(df, "cuda") if deform else None


@pytest.mark.parametrize("P,D,deform", [(1000, 16, False), (1000, 32, True), (60000, 64, True), (2000, 128, True),
                                        (60000, 256, False)])
def test_render(P, D, deform):
    W, H = 96, 64
    scene, field = _case(P, D, deform)
    cam = camera_struct(synth.make_camera(W, H, 80.0))
    rast = Rasterizer(P, D, W, H, max_dups=64 * P + 4096)
    g = [torch.randn(s, device="cuda") for s in ((3, H, W), (H, W), (H, W), (H * W, D))]
    fwd, bwd = bench.render_launches(P, D, deform)
    assert _launches(lambda: rast.forward(scene, cam, field, 0.3)) == fwd
    assert _launches(lambda: rast.backward(scene, cam, field, 0.3, *g)) == bwd


@pytest.mark.parametrize("P,D,deform,views", [(1000, 32, True, 3), (60000, 256, False, 2), (1000, 64, True, 1),
                                              (1000, 32, False, 6)])
def test_batch(P, D, deform, views):
    scene, field = _case(P, D, deform)
    W, H = 64, 48
    br = BatchRenderer(scene, field, [View(camera_struct(synth.make_camera(W, H, 60.0)), k / views,
                                           torch.rand(3, H, W, device="cuda"),
                                           torch.randn(H * W, D, device="cuda")) for k in range(views)], None)
    assert _launches(br.run) == bench.batch_launches(P, D, deform, views)


@pytest.mark.parametrize("D", [32, 128])
def test_decoder(D):
    HW = 640
    dec = Decoder(torch.randn(256, D, device="cuda").to(torch.bfloat16), torch.zeros(256, device="cuda"))
    feat, target = torch.randn(HW, D, device="cuda").to(torch.bfloat16), torch.randn(HW, 256, device="cuda")
    assert _launches(lambda: dec.l1(feat, target)) == bench.dec_launches(D) + 1
