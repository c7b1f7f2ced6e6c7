"""Lists around the sizes in which the blends stage them -- 64 entries scanned
together, a flush after more than 32 (forward) or 16 (backward) that reach the
strip, groups of three in the backward -- against the oracle, with all of a list's
Gaussians reaching the strip and with every other one beside it."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_helpers import PARAMS, assert_close_frac, assert_close_rows, gpu_forward, grads_like

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3, 4, 16, 17, 18, 31, 32, 33, 63, 64, 65, 80, 81, 96, 97, 128, 129, 195])
@pytest.mark.parametrize("every", [1, 2])
@pytest.mark.parametrize("tile", [(16, 16), (8, 8)])
def test_lists_around_the_staging_sizes(cuda_lib, n, every, tile):
    rng = np.random.default_rng(n)
    scene = synth.make_scene(n, 1, seed=n)
    vm = np.zeros((1, 3, 4), np.float32)
    vm[:, :, :3] = np.eye(3, dtype=np.float32)
    one = lambda v, t=np.float32: np.full(1, v, t)  # noqa: E731
    cams = synth.Cameras(one(16, np.int32), one(16, np.int32), one(40.0), one(40.0), one(8.0), one(8.0), vm,
                         np.zeros((1, 3), np.float32), one(0.2))
    z = 2.0 + rng.uniform(0, 1, n)
    centre = np.where((np.arange(n) % every)[:, None] == 0, rng.uniform(-3, 3, (n, 2)), [[6.0, -6.0]])  # in pixels
    scene.means[:] = np.concatenate([centre / 40.0 * z[:, None], z[:, None]], 1).astype(np.float32)
    scene.log_scales[:] = rng.uniform(-3.0, -2.6, (n, 3)).astype(np.float32)  # 1 to 1.5 pixels
    scene.opacity_logits[:] = rng.uniform(-4.0, -2.5, n).astype(np.float32)  # no pixel stops
    bg = (0.1, 0.2, 0.3)
    ref = oracle.forward(scene, cams, tile, bg=bg)
    rz, sc, params, img = gpu_forward(cuda_lib, scene, cams, tile, bg)
    amb = ref["amb"] != 0
    assert amb.mean() < 0.1
    assert_close_frac(img.cpu().numpy()[~np.tile(amb, 3)], ref["img"][~np.tile(amb, 3)], 0, 1e-4, "image")
    dimg = rng.normal(size=ref["img"].shape).astype(np.float32)
    dimg[np.tile(amb, 3)] = 0.0
    grads, _, _ = oracle.backward(scene, cams, ref, dimg.astype(np.float64), tile, bg)
    got = grads_like(params)
    rz.backward(sc, torch.tensor(dimg, device="cuda"), got)
    bad = np.zeros(n, bool)
    bad[np.nonzero(ref["P"]["amb"])[0] % n] = True
    assert bad.mean() < 0.1 or n < 10
    for k in PARAMS:
        ref_k = grads[k][~bad]
        if len(ref_k):
            assert_close_rows(got[k].cpu().numpy()[~bad], ref_k, 1e-3, 1e-5 * np.abs(ref_k).max(), k)
