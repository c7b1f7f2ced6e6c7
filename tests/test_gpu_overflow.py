"""A capturable render whose lists need more keys than there is room for shows the
background, also when the (record, bin) entries that were kept would fill the room
exactly (Gaussians of one tile each)."""
import numpy as np
import pytest
import torch

import synth
from gpu_helpers import grads_like, scene_to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("views", [1, 3])  # one bin in all; one bin per view
def test_too_few_keys_show_the_background(cuda_lib, views):
    n, side, tile, z0 = 20_000, 128, 16, 2.0
    rng = np.random.default_rng(3)
    scene = synth.make_scene(n, 0, seed=3)
    # at the centres of tiles, about a pixel wide
    f = 200.0
    cell = rng.integers(0, side // tile, (n, 2)) * tile + tile / 2
    z = z0 + 0.01 * rng.uniform(size=n)
    scene.means[:, 0], scene.means[:, 1], scene.means[:, 2] = [
        v.astype(np.float32) for v in ((cell[:, 0] - side / 2) / f * z, (cell[:, 1] - side / 2) / f * z, z)]
    scene.log_scales[:] = np.float32(-7.0)
    f32 = np.float32
    vm = np.zeros((views, 3, 4), f32)
    vm[:, :, :3] = np.eye(3, dtype=f32)
    full = lambda v, t=f32: np.full(views, v, t)  # noqa: E731
    cams = synth.Cameras(full(side, np.int32), full(side, np.int32), full(f), full(f), full(side / 2), full(side / 2),
                         vm, np.zeros((views, 3), f32), full(0.2))
    params = scene_to_device(scene)
    sc = cuda_lib.make_scene(params, 0)
    bg = (0.25, 0.5, 0.75)
    rz = cuda_lib.Rasterizer(cams, tile=(tile, tile), bg=bg, capturable=True, headroom=1.0)
    rz.reserve(n, views * n, views * n // 3)
    img = rz.forward(sc)
    grads = grads_like(params)
    rz.backward(sc, torch.ones_like(img), grads)
    torch.cuda.synchronize()
    c = rz.counts()
    assert c["records_needed"] == c["keys_needed"] == views * n > rz.cap.keys and not rz.fits()
    rec = rz.records()
    assert int(rec["ranges"].abs().max()) == 0
    want = torch.tensor(bg, device="cuda").repeat_interleave(side * side).repeat(views)
    assert torch.equal(img, want)
    assert all(int(g.count_nonzero()) == 0 for g in grads.values())
