"""The deformation module without reverse state (its MLP on the tensor
cores) against the FP64 oracle: every level count and feature width, counts
around a warp's 16 and a block's 128 Gaussians, bf16 features."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import fst as OF  # noqa: E402
from paper_2503_06161_gb300 import synth  # noqa: E402
from paper_2503_06161_gb300.fst import FSTDeform  # noqa: E402
from paper_2503_06161_gb300.raster import GaussianScene  # noqa: E402

from gpu_helpers import TOL_FEAT_REL, rel_err  # noqa: E402

LO, HI = (-2.0, -2.0, 3.0), (2.0, 2.0, 8.0)


@pytest.mark.parametrize("P,levels,D,bf16", [(1, 1, 16, False), (15, 2, 32, False), (16, 3, 64, False),
                                             (17, 4, 128, False), (127, 4, 32, True), (129, 1, 128, True),
                                             (1000, 3, 16, False), (641, 2, 64, True)])
def test_forward_only_matches_oracle(P, levels, D, bf16):
    # The bar of the training forward (1e-4 of the offsets' scale): the
    # three-term products are as exact as FP32 ones.
    rs, rt, t = 8, 6, 0.43
    sc = synth.make_scene(P, D, LO, HI, seed=P, bf16_storage=bf16)
    planes, mlp = synth.make_fst(levels, rs, rt, D, seed=P + 1, plane_std=0.2, head_std=0.5, dz_std=0.5, bias_std=0.1)
    scene = GaussianScene.from_numpy(sc, "cuda", bf16=bf16)
    fst = FSTDeform.from_numpy(planes, mlp, levels, rs, rt, D, LO, HI, P, with_backward=False)
    st = fst.forward(scene, t)
    torch.cuda.synchronize()
    feat = synth.bf16_round(sc.feat) if bf16 else sc.feat
    out = OF.forward(OF.unpack_planes(planes, levels, rs, rt), OF.unpack_mlp(mlp, levels, D),
                     np.asarray(sc.means, np.float64), t, LO, HI, levels, rs, rt)
    ref = OF.apply(sc.means, sc.quats, sc.log_scales, sc.opacity_logits, feat, out)
    canon = [sc.means, sc.quats, sc.log_scales, sc.opacity_logits, feat]
    for name, got, r, c in zip(["means", "quats", "log_scales", "logits", "feat"],
                               [st.means, st.quats, st.log_scales, st.opacity_logits, st.feat], ref, canon):
        g = got.float().cpu().numpy().astype(np.float64)
        c = np.asarray(c, np.float64).reshape(g.shape)
        r = np.asarray(r, np.float64).reshape(g.shape)
        if name == "feat" and bf16:  # rounded once on the way out
            assert np.all(np.abs(g - r) <= 2.0 ** -8 * np.abs(r) + 1e-5 * (np.abs(c) + np.abs(r - c)) + 1e-30)
        else:
            assert rel_err(g - c, r - c) < TOL_FEAT_REL, name
