"""The integer stage at the sizes where it changes form: the one-launch sort
(whole and part blocks, one to three keys a thread, its last size and the
first one of the passes), the Gaussians per block of the tile lists, and more
tiles than the narrow scatter takes.  Everything bit-exact against the
oracle; a third of the depths are ties, some Gaussians are culled."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import oracle as O  # noqa: E402

from test_gpu_render import _tile_bin_gpu  # noqa: E402


@pytest.mark.parametrize("P,W,H,tile", [
    (1, 40, 24, (16, 16)), (31, 40, 24, (32, 8)), (1023, 97, 61, (16, 16)), (1024, 97, 61, (8, 32)),
    (1025, 97, 61, (16, 16)), (2049, 97, 61, (16, 16)), (16384, 203, 157, (16, 16)), (16385, 203, 157, (16, 16)),
    (32769, 203, 157, (16, 16)), (38912, 203, 157, (16, 16)), (49152, 203, 157, (16, 16)),
    (49153, 203, 157, (16, 16)), (77823, 203, 157, (16, 16)), (77825, 203, 157, (16, 16)),
    (3000, 1100, 520, (16, 16)), (20001, 1100, 520, (16, 16)), (79000, 1100, 520, (16, 16)),
    (622591, 97, 61, (16, 16)), (622593, 203, 157, (16, 16))])
def test_tile_lists_bit_exact(P, W, H, tile):
    rng = np.random.default_rng(P)
    uv = np.c_[rng.uniform(-20, W + 20, P), rng.uniform(-20, H + 20, P)].astype(np.float32)
    radius = rng.integers(-1, 24, P).astype(np.int32)
    depth = rng.uniform(0.5, 10, P).astype(np.float32)
    tie = rng.random(P) < 0.33
    depth[tie] = np.float32(0.5) + rng.integers(0, 7, P)[tie].astype(np.float32)
    keys, gauss, ranges = _tile_bin_gpu(uv, radius, depth, W, H, tile)
    k_ref, v_ref, r_ref = O.tile_bin(uv, radius, depth, W, H, *tile)
    assert len(keys) == len(k_ref)
    assert np.array_equal(keys, k_ref)
    assert np.array_equal(gauss, v_ref)
    # A tile without entries has an empty range (the oracle's starts at 0, the
    # kernel's where the next tile starts).
    some = r_ref[:, 1] > r_ref[:, 0]
    assert np.array_equal(ranges[some], r_ref[some])
    assert np.array_equal(ranges[~some, 0], ranges[~some, 1])
