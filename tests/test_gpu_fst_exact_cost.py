"""The exact plane-gradient sums of the deformation module's reverse cost what
their documentation says: about three times the reverse with float atomics."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2503_06161_gb300 import synth  # noqa: E402
from paper_2503_06161_gb300.fst import FSTDeform  # noqa: E402
from paper_2503_06161_gb300.raster import GaussianScene  # noqa: E402

LO, HI = (-2.0, -2.0, 3.0), (2.0, 2.0, 8.0)


def _reverse_time(exact, P=50000, levels=4, rs=64, rt=100, D=32):
    planes, mlp = synth.make_fst(levels, rs, rt, D)
    scene = GaussianScene.from_numpy(synth.make_scene(P, D, LO, HI, seed=1), "cuda")
    fst = FSTDeform.from_numpy(planes, mlp, levels, rs, rt, D, LO, HI, P, exact_planes=exact)
    gen = torch.Generator(device="cuda").manual_seed(2)
    g = {k: 1e-6 * torch.randn(getattr(scene, k).shape, generator=gen, device="cuda")
         for k in ("means", "quats", "log_scales", "opacity_logits", "feat")}
    fst.forward(scene, 0.4)
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    times = []
    for _ in range(9):
        ev[0].record()
        for _ in range(4):
            fst.backward(scene, 0.4, g)
        ev[1].record()
        torch.cuda.synchronize()
        times.append(250.0 * ev[0].elapsed_time(ev[1]))
    return sorted(times[2:])[3]


def test_exact_sums_cost_about_three_times_the_reverse():
    exact, plain = _reverse_time(True), _reverse_time(False)
    # 4.8 times with four neighbouring channels to a lane, whose 8-byte atomics
    # lie 32 bytes apart; 3.1 with every eighth channel (1530 and 490 us).
    assert exact < 4.0 * plain, (exact, plain)
