"""Gaussians hundreds of pixels long and a pixel wide: their exponent is a small
difference of terms of a million, so its float32 rounding is far above 1/1000.  The
test that leaves a Gaussian out of a strip must allow for it: what a pixel blends
must not depend on the strip the pixel is in, so not on the pixels per lane."""
import numpy as np
import pytest
import torch

import synth
from gpu_helpers import PARAMS, grads_like, scene_to_device

pytestmark = pytest.mark.gpu


def _needles(n, seed, long=(-1.5, 0.7)):
    rng = np.random.default_rng(seed)
    scene = synth.make_scene(n, 0, seed=seed)
    scene.log_scales[:] = np.float32(-8.0)
    scene.log_scales[:, 0] = rng.uniform(*long, n).astype(np.float32)  # 80 to 700 pixels at distance 3
    scene.opacity_logits[:] = rng.uniform(-4.0, -1.5, n).astype(np.float32)  # few pixels stop early
    return scene


def _render(cuda_lib, sc, cams, tile, ppt):
    rz = cuda_lib.Rasterizer(cams, tile=tile, pixels_per_thread=ppt)
    img = rz.forward(sc, depth=True, stats=True)
    rec = rz.records()
    return rz, [img] + [rec[k].clone() for k in ("n_contrib", "final_T", "depth_acc", "pixel_stats")]


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_needles_blend_alike_in_every_strip(cuda_lib, seed):
    scene, cams = _needles(3000, seed), synth.make_cameras([(1264, 832), (801, 1203), (1000, 700)], radius=3.0, seed=seed)
    params = scene_to_device(scene)
    sc = cuda_lib.make_scene(params, 0)
    ref = None
    for ppt in (8, 4, 2, 1):
        _, out = _render(cuda_lib, sc, cams, (32, 64), ppt)
        if ref is None:
            ref = out
            assert int(ref[4][:, 1].sum()) > 5_000_000  # blended pairs
        differ = [int((a != b).sum()) for a, b in zip(out, ref)]
        assert differ == [0] * len(differ), ppt


def test_needles_in_a_small_render_give_the_same_gradients(cuda_lib):
    """A small render's forward takes fewer pixels per lane than its backward: the
    gradients are those of a forward in the backward's own strips."""
    scene, cams = _needles(3000, 4), synth.make_cameras([(512, 500)], radius=1.6, seed=4)
    params = scene_to_device(scene)
    sc = cuda_lib.make_scene(params, 0)
    runs = []
    for ppt in (0, 4):
        rz, out = _render(cuda_lib, sc, cams, (32, 64), ppt)
        dimg = torch.randn(out[0].shape, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
        grads = grads_like(params)
        rz.backward(sc, dimg, grads)
        runs.append((out, grads))
    for a, b in zip(runs[0][0], runs[1][0]):
        assert torch.equal(a, b)
    for k in PARAMS:  # the same kernel on the same state: only the order of its atomics may differ
        a, b = runs[0][1][k].double(), runs[1][1][k].double()
        assert float((a - b).norm()) <= 1e-5 * float(b.norm()) + 1e-12
