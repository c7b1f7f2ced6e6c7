"""The forward blend's two paths -- packed pixel pairs for plain Gaussians, pixel
by pixel with every test for the others -- and its pixel counts per lane: images
against the oracle with Gaussians of both kinds (opacities on either side of the
0.99 clamp, needles whose conic is nearly degenerate, supports that cut the
alpha >= 1/255 ellipse), bit for bit the same for 1, 2, 4 and 8 pixels per lane,
and a colour that is not finite changes only the pixels that blend it."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_helpers import PARAMS, assert_close_frac, assert_close_rows, gpu_forward, grads_like, scene_to_device

pytestmark = pytest.mark.gpu


def _mixed_scene(n, seed, needles=True):
    rng = np.random.default_rng(seed)
    sc = synth.make_scene(n, 1, seed=seed)
    kind = rng.integers(0, 4, n)
    sc.opacity_logits[kind == 0] = rng.uniform(3.0, 9.0, int((kind == 0).sum())).astype(np.float32)  # o 0.953 .. 0.9999
    needle = (kind == 1) & needles
    sc.log_scales[needle] = np.float32(-8.0)
    sc.log_scales[needle, 0] = rng.uniform(-2.0, -0.5, int(needle.sum())).astype(np.float32)
    return sc


@pytest.mark.parametrize("n,sizes", [(40, [(120, 90)]), (700, [(97, 61), (64, 128)])])
def test_plain_and_other_gaussians_match_the_oracle(cuda_lib, n, sizes):
    scene, cams = _mixed_scene(n, 100 + n), synth.make_cameras(sizes, radius=3.0, seed=5)
    ref = oracle.forward(scene, cams, (16, 16), bg=(0.1, 0.2, 0.3))
    rz, _, _, img = gpu_forward(cuda_lib, scene, cams, (16, 16), (0.1, 0.2, 0.3))
    amb = ref["amb"] != 0
    _, _, _, base = oracle.layout(cams, (16, 16))
    amb3 = np.concatenate([np.tile(amb[base[v]:base[v + 1]], 3) for v in range(cams.V)])
    assert amb.mean() < 0.1
    assert_close_frac(img.cpu().numpy()[~amb3], ref["img"][~amb3], 0, 1e-4, "image")
    assert_close_frac(rz.records()["final_T"].cpu().numpy()[~amb], ref["T"][~amb], 0, 1e-4, "final T")


@pytest.mark.parametrize("seed", [1, 2])
def test_pixels_per_lane_do_not_change_a_bit(cuda_lib, seed):
    scene, cams = _mixed_scene(3000, seed), synth.make_cameras([(203, 157), (90, 301)], radius=3.0, seed=seed)
    params = scene_to_device(scene)
    sc = cuda_lib.make_scene(params, scene.sh_degree)
    runs = []
    for ppt in (0, 1, 2, 4, 8):
        rz = cuda_lib.Rasterizer(cams, tile=(32, 64), pixels_per_thread=ppt)
        img = rz.forward(sc, depth=True, stats=True)
        rec = rz.records()
        runs.append([img] + [rec[k].clone() for k in ("final_T", "n_contrib", "depth_acc", "pixel_stats")])
        img2 = rz.forward(sc)
        assert torch.equal(img, img2)
    for r in runs[1:]:
        for a, b in zip(r, runs[0]):
            assert torch.equal(a, b)


def test_a_colour_that_is_not_finite_stays_where_it_blends(cuda_lib):
    scene, cams = synth.make_scene(400, 0, seed=9), synth.make_cameras([(150, 110)], radius=3.0, seed=9)
    params = scene_to_device(scene)
    g = int(torch.argmin((params["means"] ** 2).sum(1)))
    imgs, T = [], []
    for value in (0.5, 1.5, float("inf"), float("nan")):
        params["sh"][g] = value
        rz = cuda_lib.Rasterizer(cams, tile=(16, 16))
        imgs.append(rz.forward(cuda_lib.make_scene(params, 0)))
        T.append(rz.records()["final_T"].clone())
    apart = imgs[0] == imgs[1]  # pixels whose colour does not hold Gaussian g
    assert 0 < int((~apart).sum()) and int(apart.sum()) > 0
    for img, t in zip(imgs[2:], T[2:]):
        assert torch.equal(img[apart], imgs[0][apart])
        assert torch.equal(t, T[0])
        assert not torch.isfinite(img[~apart]).any()


@pytest.mark.parametrize("n,sizes,ppt", [(40, [(120, 90)], 0), (700, [(97, 61), (64, 128)], 0), (700, [(97, 61), (64, 128)], 1),
                                         (700, [(97, 61), (64, 128)], 2), (700, [(97, 61), (64, 128)], 8)])
def test_gradients_with_opacities_around_the_clamp_match_the_oracle(cuda_lib, n, sizes, ppt):
    # (no needles: the gradient of a nearly degenerate covariance is a float32
    # cancellation that no order of summation brings within the tolerance)
    scene, cams = _mixed_scene(n, 100 + n, needles=False), synth.make_cameras(sizes, radius=3.0, seed=5)
    tile, bg = (32, 64), (0.1, 0.2, 0.3)
    ref = oracle.forward(scene, cams, tile, bg=bg)
    amb = ref["amb"] != 0
    _, _, _, base = oracle.layout(cams, tile)
    dimg = np.random.default_rng(3).normal(size=ref["img"].shape).astype(np.float32)
    dimg[np.concatenate([np.tile(amb[base[v]:base[v + 1]], 3) for v in range(cams.V)])] = 0.0
    grads, _, _ = oracle.backward(scene, cams, ref, dimg.astype(np.float64), tile, bg)
    params = scene_to_device(scene)
    sc = cuda_lib.make_scene(params, scene.sh_degree)
    rz = cuda_lib.Rasterizer(cams, tile=tile, bg=bg, pixels_per_thread=ppt)
    rz.forward(sc)
    got = grads_like(params)
    rz.backward(sc, torch.tensor(dimg, device="cuda"), got)
    bad = np.zeros(scene.n, bool)
    bad[np.nonzero(ref["P"]["amb"])[0] % scene.n] = True
    for k in PARAMS:
        ref_k = grads[k][~bad]
        assert_close_rows(got[k].cpu().numpy()[~bad], ref_k, 1e-3, 1e-5 * np.abs(ref_k).max(), k)


@pytest.mark.parametrize("value", [float("nan"), float("inf"), 1e30])
def test_a_pixel_gradient_reaches_only_the_gaussians_it_blends(cuda_lib, value):
    scene, cams = synth.make_scene(400, 0, seed=9), synth.make_cameras([(150, 110)], radius=3.0, seed=9)
    params = scene_to_device(scene)
    sc = cuda_lib.make_scene(params, 0)
    rz = cuda_lib.Rasterizer(cams, tile=(16, 16))
    img = rz.forward(sc)
    pixel = 55 * 150 + 75
    one = torch.zeros_like(img)
    one[pixel] = 1.0
    base = torch.randn(img.shape, device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    base[pixel] = 0.0
    runs = []
    for dimg in (one, base, torch.where(one > 0, torch.full_like(base, value), base)):
        g = grads_like(params)
        rz.backward(sc, dimg, g)
        runs.append(g)
    apart = (runs[0]["sh"].reshape(scene.n, -1) == 0).all(1)  # not blended at the pixel
    assert 0 < int((~apart).sum()) < scene.n
    for k in PARAMS:
        a, b = runs[1][k][apart], runs[2][k][apart]
        assert torch.isfinite(b).all(), k
        torch.testing.assert_close(b, a, rtol=1e-4, atol=1e-6 * float(a.abs().max()))


@pytest.mark.parametrize("tile,size", [((16, 16), (512, 512)), ((16, 16), (528, 512)), ((32, 64), (960, 960)),
                                       ((32, 64), (960, 1024)), ((8, 8), (512, 512))])
def test_small_renders_choose_pixels_per_lane_freely(cuda_lib, tile, size):
    scene, cams = _mixed_scene(2000, 9), synth.make_cameras([size], radius=3.0, seed=2)
    params = scene_to_device(scene)
    sc = cuda_lib.make_scene(params, scene.sh_degree)
    # strips of 8 columns and 4 rows per pixel of a lane
    most = min(4, tile[1] // 4)
    runs = []
    for ppt in (0, most):
        rz = cuda_lib.Rasterizer(cams, tile=tile, pixels_per_thread=ppt)
        img = rz.forward(sc, depth=True, stats=True)
        rec = rz.records()
        grads = grads_like(params)
        rz.backward(sc, torch.ones_like(img), grads)
        runs.append(([img] + [rec[k].clone() for k in ("final_T", "n_contrib", "depth_acc", "pixel_stats")], grads))
    for a, b in zip(runs[0][0], runs[1][0]):
        assert torch.equal(a, b)
    for k in PARAMS:  # the same kernel on the same state: only the order of its atomics may differ
        a, b = runs[0][1][k].double(), runs[1][1][k].double()
        assert float((a - b).norm()) <= 1e-5 * float(b.norm()) + 1e-12


@pytest.mark.parametrize("tile,size", [((16, 16), (70, 53)), ((32, 64), (96, 128)), ((8, 8), (64, 64))])
def test_both_backward_paths_round_alike(cuda_lib, tile, size):
    """An enormous gradient on pixels that no Gaussian reaches sends their strips to
    the general path: the conic gradients (summed in double precision) keep every bit."""
    scene = synth.make_scene(150, 1, seed=3)
    scene.log_scales[:] -= np.float32(0.5)
    cams = synth.make_cameras([size], radius=5.0, seed=4)
    params = scene_to_device(scene)
    sc = cuda_lib.make_scene(params, scene.sh_degree)
    rz = cuda_lib.Rasterizer(cams, tile=tile)
    img = rz.forward(sc)
    idle = rz.records()["n_contrib"].flatten() == 0
    assert 0 < int(idle.sum()) < idle.numel()
    dimg = torch.randn(img.numel(), device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    dimg[idle.repeat(3)] = 0.0
    runs = []
    for value in (0.0, 1e26):
        d = torch.where(idle.repeat(3), torch.full_like(dimg, value), dimg).reshape(img.shape)
        grads = grads_like(params)
        rz.backward(sc, d.contiguous(), grads)
        runs.append(grads)
    for k in ("log_scales", "quats"):
        assert torch.equal(runs[0][k], runs[1][k]), k
