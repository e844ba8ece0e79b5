"""Plane and plane-gradient arrays of the deformation module that are not
16-byte aligned (a view into a larger buffer)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import fst as OF  # noqa: E402
from paper_2503_06161_gb300 import _lib, synth  # noqa: E402
from paper_2503_06161_gb300.fst import FSTDeform  # noqa: E402
from paper_2503_06161_gb300.raster import GaussianScene  # noqa: E402

from gpu_helpers import rel_err  # noqa: E402

LO, HI = (-2.0, -2.0, 3.0), (2.0, 2.0, 8.0)


def _view(x, skew):
    """A copy of x at 4 skew bytes into a NaN-filled buffer."""
    store = torch.full((x.numel() + 8,), float("nan"), device="cuda")
    store[skew:skew + x.numel()] = x
    return store, store[skew:skew + x.numel()]


def _case(P, levels, rs, rt, D, exact):
    sc = synth.make_scene(P, D, LO, HI, seed=3)
    planes, mlp = synth.make_fst(levels, rs, rt, D, seed=4, plane_std=0.2, head_std=0.5, dz_std=0.5, bias_std=0.1)
    scene = GaussianScene.from_numpy(sc, "cuda")
    fst = FSTDeform.from_numpy(planes, mlp, levels, rs, rt, D, LO, HI, P, exact_planes=exact)
    gen = torch.Generator(device="cuda").manual_seed(6)
    g = {k: torch.randn(getattr(scene, k).shape, generator=gen, device="cuda")
         for k in ("means", "quats", "log_scales", "opacity_logits", "feat")}
    return scene, fst, g


@pytest.mark.parametrize("exact", [True, False])
@pytest.mark.parametrize("P,levels,D,skew_p,skew_d", [(300, 4, 32, 1, 0), (37, 2, 16, 2, 0), (129, 1, 64, 3, 1)])
def test_reverse_takes_unaligned_planes(P, levels, D, skew_p, skew_d, exact):
    rs, rt, t = 6, 5, 0.61
    scene, fst, g = _case(P, levels, rs, rt, D, exact)
    fst.forward(scene, t)

    def reverse(planes, d_planes):
        st = _lib.make_fst(levels, rs, rt, D, planes, fst.mlp, LO, HI, exact)
        d_means, d_mlp = torch.empty(P, 3, device="cuda"), torch.empty_like(fst.mlp)
        _lib.fe_fst_backward(st, P, scene.means, t, g["means"], g["quats"], g["log_scales"], g["opacity_logits"],
                             g["feat"], d_means, d_planes, d_mlp, fst.workspace)
        torch.cuda.synchronize()
        return [x.cpu().numpy().astype(np.float64) for x in (d_means, d_planes, d_mlp)]

    want = reverse(fst.planes, torch.empty_like(fst.planes))
    _, planes = _view(fst.planes, skew_p)
    store, d_planes = _view(torch.zeros_like(fst.planes), skew_d)
    got = reverse(planes, d_planes)
    assert torch.isnan(store[:skew_d]).all() and torch.isnan(store[skew_d + d_planes.numel():]).all()
    assert np.array_equal(got[2], want[2])
    # Sums over channels (means) and, unless exact, over Gaussians (planes) in
    # another order: at most a few hundred float32 roundings each.
    assert rel_err(got[0], want[0]) < 1e-4
    if exact:
        assert np.array_equal(got[1], want[1])
    else:
        assert rel_err(got[1], want[1]) < 1e-4


@pytest.mark.parametrize("skew_p,skew_d", [(0, 1), (3, 0), (2, 2)])
def test_total_variation_takes_unaligned_arrays(skew_p, skew_d):
    # The reverse's gradient array may be unaligned, and the TV term is added
    # to that same array.  Same sums in the same order: same bits.
    levels, rs, rt, D = 2, 6, 5, 16
    _, fst, _ = _case(1, levels, rs, rt, D, False)
    base = torch.randn(fst.planes.numel(), generator=torch.Generator(device="cuda").manual_seed(8), device="cuda")

    def tv(planes, d_planes):
        loss, scratch = torch.zeros(1, device="cuda"), torch.empty(1024, device="cuda")
        _lib.fe_fst_tv(_lib.make_fst(levels, rs, rt, D, planes, fst.mlp, LO, HI), 0.7, loss, d_planes, scratch)
        torch.cuda.synchronize()
        return loss.item(), d_planes.clone()

    want = tv(fst.planes, base.clone())
    store, d_planes = _view(base, skew_d)
    got = tv(_view(fst.planes, skew_p)[1], d_planes)
    assert got[0] == want[0]
    assert torch.equal(got[1], want[1])
    assert torch.isnan(store[:skew_d]).all() and torch.isnan(store[skew_d + d_planes.numel():]).all()
