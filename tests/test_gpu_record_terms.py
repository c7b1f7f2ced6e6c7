"""Preprocessing and its backward over view counts on both sides of their lane
groups and camera tables (2, 4 and 8 lanes per Gaussian, by record up to 8
views, views in shared memory from 7, 32 per table), warps that are
not full, every SH degree and SH rows that are not 16-byte aligned: a render of
V views against V renders of one view."""
import pytest
import torch

import synth
from gpu_helpers import grads_like, scene_to_device

pytestmark = pytest.mark.gpu


def _run(mvgs, params, degree, cams, seed, grads=None):
    sc = mvgs.make_scene(params, degree)
    rz = mvgs.Rasterizer(cams, tile=(16, 16))
    img = rz.forward(sc)
    g = torch.Generator("cuda").manual_seed(seed)
    dimg = torch.randn(img.shape, device="cuda", generator=g)
    grads = grads_like(params) if grads is None else grads
    for t in grads.values():
        t.fill_(float("nan"))
    rec = {k: v.clone() for k, v in rz.records().items()}
    r = rec["g"].shape[0]
    m2d, e1 = torch.empty(r, 2, device="cuda"), torch.empty(r, device="cuda")
    rz.backward(sc, dimg, grads, m2d, e1)
    return img, dimg, grads, rec, m2d, e1, (sc, rz)


def _rel(a, b):
    a, b = a.double(), b.double()
    return float((a - b).norm() / b.norm().clamp_min(1e-30))


# Both sides form the same per-record terms.  The blend backward adds a record's
# pixels in an order that may vary (float32: some 1e-7 of the result for these
# few pixels), and the sums over V terms differ by less than V 2^-24 = 2e-6 of
# their size; 1e-5 of the tensor's norm covers both.
@pytest.mark.parametrize("V", [1, 2, 3, 4, 5, 7, 8, 9, 33, 40])
@pytest.mark.parametrize("n,degree", [(1, 3), (31, 2), (64, 0), (97, 1), (200, 3)])
def test_views_at_once_equal_views_one_by_one(cuda_lib, V, n, degree):
    scene = synth.make_scene(n, degree, seed=n)
    cams = synth.make_cameras([(40 + 3 * (v % 5), 30 + v % 7) for v in range(V)], radius=3.0, seed=V)
    params = scene_to_device(scene)
    img, dimg, grads, rec, m2d, e1, _ = _run(cuda_lib, params, degree, cams, 7)
    total = {k: torch.zeros_like(v, dtype=torch.float64) for k, v in params.items()}
    at = 0
    for v in range(V):
        one = cams.subset([v])
        sc = cuda_lib.make_scene(params, degree)
        rz = cuda_lib.Rasterizer(one, tile=(16, 16))
        im = rz.forward(sc)
        part = slice(at, at + im.numel())
        at += im.numel()
        assert torch.equal(im.flatten(), img.flatten()[part])
        ids = rz.records()["g"].clone()
        g1 = grads_like(params)
        m1, f1 = torch.empty(ids.shape[0], 2, device="cuda"), torch.empty(ids.shape[0], device="cuda")
        rz.backward(sc, dimg.flatten()[part].reshape(im.shape).contiguous(), g1, m1, f1)
        for k in total:
            total[k] += g1[k].double()
        mine = rec["v"] == v
        assert torch.equal(rec["g"][mine], ids)
        if ids.numel():
            assert _rel(m2d[mine], m1) <= 1e-5 and _rel(e1[mine], f1) <= 1e-5
    for k, g in grads.items():
        assert torch.isfinite(g).all()
        assert _rel(g, total[k]) <= 1e-5, k


@pytest.mark.parametrize("V,degree", [(1, 1), (3, 3), (8, 3), (8, 0), (34, 1)])
def test_unaligned_sh_rows(cuda_lib, V, degree):
    scene = synth.make_scene(150, degree, seed=3)
    cams = synth.make_cameras([(45, 37)] * V, radius=3.0, seed=V)
    params = scene_to_device(scene)
    img, _, grads, *_ = _run(cuda_lib, params, degree, cams, 5)

    def shifted(t):
        s = torch.empty(t.numel() + 1, device="cuda")[1:].view(t.shape)
        return s.copy_(t)

    moved = dict(params, sh=shifted(params["sh"]))
    out = dict(grads_like(params), sh=shifted(params["sh"]))
    img2, _, grads2, *_ = _run(cuda_lib, moved, degree, cams, 5, out)
    assert torch.equal(img, img2)
    for k in grads:
        assert _rel(grads2[k], grads[k]) <= 1e-5, k
