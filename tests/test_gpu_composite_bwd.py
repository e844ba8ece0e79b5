"""The reverse compositing's chunks of a warp's entries, against the FP64
oracle: batches whose every entry is blended by every warp (the most entries
a warp can hold), batches of few entries, alphas at the clamp, ragged images
and every tile shape and pass width."""
import dataclasses

import numpy as np
import pytest

from oracle import oracle as O
from paper_2503_06161_gb300 import synth
from tests.gpu_helpers import check_forward, check_grads, forward_parity, gpu_backward, gpu_forward, grad_parity

pytestmark = pytest.mark.gpu


def _thick_scene(P, D, seed):
    """Faint Gaussians that cover the whole image (every pixel blends every
    one of them), every ninth a small one whose centre is past the clamp."""
    sc = synth.make_scene(P, D, (-0.3, -0.3, 3.0), (0.3, 0.3, 8.0), seed=seed)
    ls, lg = sc.log_scales.copy(), sc.opacity_logits.copy()
    ls += 3.5
    lg[:] = -3.5 + 0.2 * lg
    ls[::9] -= 5.0
    lg[::9] = 6.0
    return dataclasses.replace(sc, log_scales=ls, opacity_logits=lg)


@pytest.mark.parametrize("P,D,W,H,tile,bf16", [(70, 16, 40, 24, (16, 16), False), (101, 32, 45, 27, (16, 16), False),
                                               (101, 32, 45, 27, (32, 8), True), (70, 64, 33, 40, (8, 32), False),
                                               (33, 128, 40, 24, (16, 16), False), (64, 64, 40, 24, (16, 16), True),
                                               (3, 32, 17, 9, (16, 16), False)])
def test_every_entry_blended_in_every_warp(P, D, W, H, tile, bf16):
    # The bar of every reverse test (1e-3 of each array's rms): the sums of
    # three-term products differ from FP32 ones by a few 2^-24.
    sc = _thick_scene(P, D, seed=3)
    if bf16:
        sc = dataclasses.replace(sc, sh=synth.bf16_round(sc.sh), feat=synth.bf16_round(sc.feat))
    cam = synth.make_camera(W, H, 0.9 * W)
    bg = (0.2, 0.1, 0.3)
    run = gpu_forward(sc, cam, tile=tile, bg=bg, bf16=bf16)
    pix = O.all_pixels(W, H)
    e, rep, flip = forward_parity(run, sc, cam, bg=bg)
    check_forward(e, rep, flagged_max=W * H)
    rng = np.random.default_rng(1)
    G = dict(rgb=rng.normal(size=(W * H, 3)), depth=0.1 * rng.normal(size=W * H), alpha=rng.normal(size=W * H),
             feat=rng.normal(size=(W * H, D)))
    got = gpu_backward(run, 0.0, G["rgb"], G["depth"], G["alpha"], G["feat"])
    errs, grep = grad_parity(got, sc, cam, None, 0.0, bg, pix, G, flip)
    check_grads(errs, grep)
