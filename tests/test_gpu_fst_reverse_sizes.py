"""The deformation module's reverse around the sizes of its tiles (16
Gaussians a warp, 128 a block, a second round of a block), every level count
and feature width, times on and between the time nodes, and a plane-gradient
array that is not 16-byte aligned, against the FP64 oracle with the bar of the
other reverse tests (1e-3 of each array's rms: sums of three-term products
and sums in another order differ from FP32 ones by a few 2^-24)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import fst as OF  # noqa: E402
from paper_2503_06161_gb300 import _lib  # noqa: E402

from gpu_helpers import TOL_GRAD_REL, rel_err  # noqa: E402
from test_gpu_fst import CELL_MARGIN, RELU_MARGIN, _case, _oracle_forward, _upstream  # noqa: E402


@pytest.mark.parametrize("P,levels,rs,rt,D,t,skew", [
    (1, 1, 6, 5, 32, 0.37, 0), (15, 2, 6, 5, 16, 0.0, 0), (16, 3, 6, 5, 64, 1.0, 0), (17, 4, 6, 5, 128, 0.5, 1),
    (127, 4, 6, 2, 32, 0.61, 0), (128, 3, 6, 5, 16, 0.61, 2), (129, 2, 6, 5, 128, 0.25, 3), (300, 1, 6, 5, 64, 0.8, 1),
    (38913, 1, 8, 5, 16, 0.61, 0)])
def test_reverse_matches_oracle(P, levels, rs, rt, D, t, skew):
    sc, scene, fst, pl, ly = _case(P, levels, rs, rt, D, seed=11)
    fst.forward(scene, t)
    out, _ = _oracle_forward(sc, pl, ly, t, levels, rs, rt, False)
    # The time is the same for all and is not differentiated, so only the
    # ReLUs and the spatial cells are decisions; a Gaussian near one of them
    # gets no upstream gradient.
    drop = OF.margins(out["state"])[0] < RELU_MARGIN
    for lv in range(levels):
        x = (out["state"]["coord"][:, :3] + 1.0) * 0.5 * ((rs << lv) - 1)
        drop |= np.abs(x - np.round(x)).min(axis=1) < CELL_MARGIN
    assert drop.sum() < 0.1 * P or P < 20
    up = _upstream(P, D, seed=P)
    for k in up:
        up[k][drop] = 0.0
    dev = {k: torch.tensor(v, dtype=torch.float32, device="cuda").contiguous() for k, v in up.items()}
    d_means = torch.empty(P, 3, device="cuda")
    store = torch.full((fst.d_planes.numel() + 8,), float("nan"), device="cuda")
    d_planes = store[skew:skew + fst.d_planes.numel()]
    d_mlp = torch.empty_like(fst.d_mlp)
    _lib.fe_fst_backward(fst.struct(), P, scene.means, t, dev["means"], dev["quats"], dev["log_scales"],
                         dev["opacity_logits"], dev["feat"], d_means, d_planes, d_mlp, fst.workspace)
    torch.cuda.synchronize()
    assert torch.isnan(store[:skew]).all() and torch.isnan(store[skew + d_planes.numel():]).all()
    ref = OF.backward(pl, ly, out["state"], up["means"], up["quats"], up["log_scales"], up["opacity_logits"],
                      up["feat"])
    assert rel_err(d_means.cpu().numpy().astype(np.float64), up["means"] + ref["mu"]) < TOL_GRAD_REL
    got_pl = d_planes.cpu().numpy().astype(np.float64)
    ref_pl = np.concatenate([x.ravel() for x in ref["planes"]])
    assert rel_err(got_pl, ref_pl) < TOL_GRAD_REL
    assert np.all(got_pl[ref_pl == 0.0] == 0.0)
    got_w = d_mlp.cpu().numpy().astype(np.float64)
    off = 0
    for j, (dw, db) in enumerate(ref["layers"]):
        assert rel_err(got_w[off:off + dw.size], dw.ravel()) < TOL_GRAD_REL, (j, "weight")
        off += dw.size
        assert rel_err(got_w[off:off + db.size], db) < TOL_GRAD_REL, (j, "bias")
        off += db.size
    assert off == got_w.size
