"""The deformation module without reverse state on values outside the range
of its three-term products (infinities, and magnitudes that round to one in
BF16): the Gaussians they reach get what FP32 products give, bit for bit the
training forward's outputs, and the others keep theirs."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import fst as OF  # noqa: E402
from paper_2503_06161_gb300 import _lib, synth  # noqa: E402
from paper_2503_06161_gb300.fst import FSTDeform  # noqa: E402
from paper_2503_06161_gb300.raster import GaussianScene  # noqa: E402

LO, HI = (-2.0, -2.0, 3.0), (2.0, 2.0, 8.0)
FIELDS = ("means", "quats", "log_scales", "opacity_logits", "feat")


def _run(planes, mlp, sc, levels, rs, rt, D, bf16, train):
    scene = GaussianScene.from_numpy(sc, "cuda", bf16=bf16)
    fst = FSTDeform.from_numpy(planes, mlp, levels, rs, rt, D, LO, HI, sc.P, with_backward=train)
    o = fst.forward(scene, 0.43)
    torch.cuda.synchronize()
    return {k: getattr(o, k).float().cpu().numpy().reshape(sc.P, -1) for k in FIELDS}


@pytest.mark.parametrize("P,levels,D,bf16,where,value", [
    (300, 4, 32, False, "plane", np.inf), (300, 2, 128, True, "plane", -np.inf), (129, 1, 16, False, "plane", np.nan),
    (300, 3, 64, False, "plane", 3.4e38), (1, 4, 32, False, "plane", np.inf), (300, 4, 32, False, "plane", 1e30),
    (200, 4, 32, False, "hidden", np.inf), (200, 2, 16, False, "branch", 3.4e38), (200, 4, 128, False, "feature", -np.inf),
    (200, 1, 64, True, "head", np.inf)])
def test_forward_only_diverges_as_training_does(P, levels, D, bf16, where, value):
    rs, rt = 8, 6
    sc = synth.make_scene(P, D, LO, HI, seed=P, bf16_storage=bf16)
    planes, mlp = synth.make_fst(levels, rs, rt, D, seed=5, plane_std=0.2, head_std=0.5, dz_std=0.5, bias_std=0.1)
    planes, mlp = np.array(planes, np.float32), np.array(mlp, np.float32)
    if where == "plane":  # a block of the first level's xy plane
        planes[:rs * rs * 32].reshape(rs, rs, 32)[2:4, 3:6, ::5] = value
    else:
        sizes = [o * i + o for o, i in OF.layer_shapes(levels, D)]
        layer = dict(hidden=4, branch=8 + 3 + 1, head=8 + 2, feature=21)[where]
        mlp[sum(sizes[:layer]) + 7] = value
    want = _run(planes, mlp, sc, levels, rs, rt, D, bf16, train=True)
    got = _run(planes, mlp, sc, levels, rs, rt, D, bf16, train=False)
    for k in FIELDS:
        out = ~(np.isfinite(want[k]) & np.isfinite(got[k]))
        assert np.array_equal(got[k][out], want[k][out], equal_nan=True), k
        # Elsewhere the bar of the forward tests, of each Gaussian's scale.
        with np.errstate(over="ignore", invalid="ignore"):
            scale = 1.0 + np.abs(np.where(np.isfinite(want[k]), want[k], 0.0)).max(axis=1, keepdims=True)
            err = np.where(out, 0.0, np.abs(got[k] - want[k]))
        assert (err <= (2.0 ** -7 if bf16 and k == "feat" else 1e-4) * scale).all(), k
