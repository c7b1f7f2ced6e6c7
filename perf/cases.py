"""What users of the multi-view Gaussian-splatting rasterizer have it do, as timed cases.

A case is a dict of plain values.  Its "kind" names the call:

  autograd   one differentiable render through autograd.render, an L1 loss on
             the images and its backward to the five parameter tensors
  train      one full-render training iteration: Rasterizer.forward,
             dssim_loss, Rasterizer.backward with the per-record outputs, and
             adc_accumulate into this iteration's statistics
  partial    one partially rendered iteration: sample_set, the sampled forward
             with depth, merge_views, dssim3d_loss, split_merged_grad, the
             sampled backward, adc_accumulate
  render     forward only: a resident scene rendered for a batch of cameras
             (set_cameras + forward, what a server does per batch and a viewer
             per frame)
  loss       dssim_loss with its gradient, by itself
  loss3d     dssim3d_loss with its gradient, by itself
  adam       adam_step on the five parameter groups of a scene
  densify    one densification step with the optimiser moments carried along

Scenes, cameras and targets follow the repository's synthetic workloads (means
U[-1,1]^3, log-scales N(-3, 0.5), opacity logits N(0, 1), cameras on a sphere
around the origin, 60 degrees of horizontal field of view, targets U[0, 1]),
drawn from the seed.  Buffers are what a user's program keeps: the rasterizer's
state and workspace sized by its own pre-count, gradient tensors, loss
workspace.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2506_12727_gb300 import autograd, mvgs

PARAMS = ("means", "log_scales", "quats", "opacity_logits", "sh")
MIXED_8 = "1264x832,1920x1080,1600x1067,1264x832,800x600,1920x1080,1264x832,1600x1067"
LAMBDA = 0.2


def listed():
    return [
        # The smallest call: one 128x128 view of 10k Gaussians, forward and
        # backward, where launches and host latency count.
        dict(name="single_10k_128", kind="autograd", n=10_000, sh=0, views="128x128", tile="16x16", batch=0, radius=3.0),
        # A small ragged iteration at the default tile: odd image sides, SH
        # degree 1, views of different sizes (a coarse stage or a test scene).
        dict(name="ragged_20k_3views", kind="train", n=20_011, sh=1, views="203x157,320x240,97x301", tile="16x16",
             batch=0, radius=4.0),
        # The ordinary training iteration: 500k Gaussians, four views, at the
        # tile and batch the autotuner picks for it.
        dict(name="train_500k_4views", kind="train", n=500_000, sh=3, views=",".join(["1264x832"] * 4), tile="32x64",
             batch=64, radius=4.0),
        # The largest training iteration: 3M Gaussians, eight views of mixed
        # resolutions, autotuned tile and batch.
        dict(name="train_3m_8views", kind="train", n=3_000_000, sh=3, views=MIXED_8, tile="32x64", batch=64,
             radius=4.0),
        # Differentiation at scale through autograd: 1M Gaussians, 16 views.
        dict(name="autograd_1m_16views", kind="autograd", n=1_000_000, sh=3, views=",".join(["1024x768"] * 16),
             tile="16x64", batch=0, radius=4.0),
        # A serving batch: a resident 2M scene, requests of mixed resolutions
        # batched into one call at the serving tile.
        dict(name="serve_2m_5views", kind="render", n=2_000_000, sh=3,
             views="640x480,1280x720,1920x1080,1280x720,640x480", tile="16x64", batch=0, radius=4.0),
        # One viewer frame at the rasterizer's default tile.
        dict(name="frame_500k_1view", kind="render", n=500_000, sh=3, views="1264x832", tile="16x16", batch=0,
             radius=4.0),
        # A partially rendered iteration at the trainer's default tile: one
        # image's worth of pixels over four views.
        dict(name="partial_500k_4views", kind="partial", n=500_000, sh=3, views=",".join(["1264x832"] * 4),
             tile="16x16", batch=0, radius=4.0),
        # The photometric loss of the largest iteration's eight images.
        dict(name="loss_8views", kind="loss", views=MIXED_8),
        # The 3D distance-aware loss of one merged image.
        dict(name="loss3d_1264x832", kind="loss3d", views="1264x832"),
        # The optimiser update of 3M SH-3 Gaussians.
        dict(name="adam_3m", kind="adam", n=3_000_000, sh=3),
        # One densification step of 1M Gaussians.
        dict(name="densify_1m", kind="densify", n=1_000_000, sh=3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sizes(views):
    return [tuple(int(x) for x in v.split("x")) for v in views.split(",")]


def _entries(c):
    """About how many (record, tile) entries a render case sorts."""
    tw, th = (int(x) for x in c["tile"].split("x"))
    per = [(1 + 0.0870 * w / tw) * (1 + 0.0870 * w / th) for w, _ in _sizes(c["views"])]
    return c["n"] * sum(per)


def draw(rng):
    kind = rng.choice(["autograd", "train", "train", "train", "render", "render", "partial", "loss", "loss3d", "adam",
                       "densify"])
    if kind == "adam":
        return dict(kind=kind, n=_log(rng, 1_000, 3_000_000), sh=rng.randrange(4))
    if kind == "densify":
        return dict(kind=kind, n=_log(rng, 1_000, 2_000_000), sh=rng.randrange(4))

    def view():
        w = _log(rng, 97, 1920)
        return "%dx%d" % (w, max(64, int(w * rng.uniform(0.55, 0.8))))

    if kind == "loss":
        return dict(kind=kind, views=",".join(view() for _ in range(rng.randint(1, 8))))
    if kind == "loss3d":
        return dict(kind=kind, views=view())
    while True:
        c = dict(kind=kind, n=_log(rng, 5_000, 3_000_000), sh=rng.randrange(4))
        if kind == "partial":  # the views of a group share a resolution
            c["views"] = ",".join([view()] * rng.randint(2, 8))
        else:
            c["views"] = ",".join(view() for _ in range(rng.randint(1, 12)))
        c["tile"] = rng.choice(["16x16", "16x16", "16x32", "16x64", "32x64", "32x64"])
        c["batch"] = rng.choice([0, 0, 64])
        c["radius"] = round(rng.uniform(3.0, 5.0), 2)
        pixels = sum(w * h for w, h in _sizes(c["views"]))
        if c["n"] > 8 * min(w * h for w, h in _sizes(c["views"])):  # a scene this fine is not seen through so few pixels
            continue
        if c["n"] * len(_sizes(c["views"])) <= 24_000_000 and _entries(c) <= 3.5e8 and pixels <= 11_000_000:
            return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed, k):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 16 + k)


def _scene(n, sh, seed):
    g = _gen(seed, 0)

    def randn(*s):
        return torch.randn(*s, device="cuda", generator=g)

    def rand(*s):
        return torch.rand(*s, device="cuda", generator=g)

    q = randn(n, 4)
    k = (sh + 1) ** 2
    coef = torch.empty(n, k, 3, device="cuda")
    if sh == 0:
        coef[:, 0] = (rand(n, 3) - 0.5) * (2.0 * math.sqrt(math.pi))
    else:
        coef[:, 0] = rand(n, 3)
        coef[:, 1:] = 0.05 * randn(n, k - 1, 3)
    return dict(means=2.0 * rand(n, 3) - 1.0, log_scales=-3.0 + 0.5 * randn(n, 3),
                quats=q / q.norm(dim=1, keepdim=True), opacity_logits=randn(n), sh=coef)


def _cameras(views, radius, seed):
    rng = np.random.default_rng([7, int(seed)])
    size = _sizes(views)
    V = len(size)
    W = np.array([s[0] for s in size], np.int32)
    H = np.array([s[1] for s in size], np.int32)
    f = (W / 2.0) / math.tan(math.radians(30.0))
    vm, pos = np.zeros((V, 3, 4)), np.zeros((V, 3))
    for v in range(V):
        d = rng.normal(size=3)
        eye = d / np.linalg.norm(d) * radius
        z = -eye / np.linalg.norm(eye)
        up = np.array([0.0, 1.0, 0.0]) if abs(z[1]) < 0.999 else np.array([0.0, 0.0, 1.0])
        x = np.cross(z, up)
        x /= np.linalg.norm(x)
        R = np.stack([x, np.cross(z, x), z])
        vm[v], pos[v] = np.concatenate([R, (-R @ eye)[:, None]], 1), eye
    f32 = np.float32
    return SimpleNamespace(V=V, width=W, height=H, fx=f.astype(f32), fy=f.astype(f32), cx=(W / 2.0).astype(f32),
                           cy=(H / 2.0).astype(f32), viewmat=vm.astype(f32), campos=pos.astype(f32),
                           near=np.full(V, 0.2, f32))


def _pixels(views):
    return sum(w * h for w, h in _sizes(views))


def _smooth(h, w, ch, g):
    """A smooth random field in [0, 1] with a little noise: what an image looks like to a window of 11 pixels."""
    low = torch.rand(1, ch, max(2, h // 16), max(2, w // 16), device="cuda", generator=g)
    x = torch.nn.functional.interpolate(low, size=(h, w), mode="bilinear", align_corners=True)[0]
    return (0.9 * x + 0.1 * torch.rand(ch, h, w, device="cuda", generator=g)).contiguous()


def _image_pair(views, seed):
    """A target image per view and a reconstruction near it, packed."""
    g = _gen(seed, 1)
    tgt = [_smooth(h, w, 3, g) for w, h in _sizes(views)]
    img = [(t + 0.1 * torch.randn(t.shape, device="cuda", generator=g)).clamp(0.0, 1.0) for t in tgt]
    return torch.cat([i.reshape(-1) for i in img]), torch.cat([t.reshape(-1) for t in tgt])


def _surface(views, seed):
    """Surface points and kernel widths of a merged image: a smooth depth map with steps, pixels lifted through a
    60-degree camera, one pixel in 50 without a surface point."""
    g = _gen(seed, 2)
    (w, h), = _sizes(views)
    f = (w / 2.0) / math.tan(math.radians(30.0))
    z = 3.0 + _smooth(h, w, 1, g)[0] + 0.5 * (_smooth(h, w, 1, g)[0] > 0.5)
    x = (torch.arange(w, device="cuda") + 0.5 - w / 2.0) / f
    y = (torch.arange(h, device="cuda") + 0.5 - h / 2.0) / f
    some = torch.rand(h, w, device="cuda", generator=g) > 0.02
    pts = torch.stack([z * x, z * y[:, None], z]) * some
    return pts.reshape(-1).contiguous(), (1.5 * z / f * some).reshape(-1).contiguous()


def _targets(views, seed):
    return torch.rand(3 * _pixels(views), device="cuda", generator=_gen(seed, 3))


def _densify_inputs(case, seed):
    """4% of the Gaussians are pruned, 10% split, 14% cloned (which ones, and by how much, is random)."""
    p = _scene(case["n"], case["sh"], seed)
    g, n = _gen(seed, 4), case["n"]
    split, clone, prune, extent = 2e-4, 2e-4, math.log(0.02 / 0.98), -2.0
    rank = torch.empty(n, dtype=torch.int64, device="cuda")
    rank[torch.randperm(n, device="cuda", generator=g)] = torch.arange(n, device="cuda")
    pruned, parted, cloned = rank < n // 25, (rank >= n // 25) & (rank < n // 7), (rank >= n // 7) & (rank < n // 7 * 2)
    far = 0.01 + torch.rand(n, device="cuda", generator=g)
    p["opacity_logits"] = torch.where(pruned, prune - far, prune + 3.0 * far)
    big = (rank % 3 == 0) & ~cloned | parted  # some large Gaussians stay as they are
    p["log_scales"][:, 0] = torch.where(big, extent + far, extent - far)
    p["log_scales"][:, 1:].clamp_(max=extent - 0.01)
    denom = torch.randint(1, 9, (n,), device="cuda", generator=g).float()
    e1 = denom * split * torch.where(parted, 1.0 + far, 1.0 / (1.0 + far))
    e2 = denom * clone * torch.where(cloned, 1.0 + far, 1.0 / (1.0 + far))
    normals = torch.randn(n, 2, 3, device="cuda", generator=g)
    carry = [0.01 * torch.randn(p[k].shape, device="cuda", generator=g) for k in PARAMS]
    carry += [1e-4 * torch.rand(p[k].shape, device="cuda", generator=g) for k in PARAMS]
    return p, e1, e2, denom, normals, carry, (split, clone, prune, extent)


def _adam_inputs(case, seed):
    p = _scene(case["n"], case["sh"], seed)
    g = _gen(seed, 5)
    grad = {k: 1e-3 * torch.randn(p[k].shape, device="cuda", generator=g) for k in PARAMS}
    m = {k: 1e-3 * torch.randn(p[k].shape, device="cuda", generator=g) for k in PARAMS}
    v = {k: 1e-6 * torch.rand(p[k].shape, device="cuda", generator=g) for k in PARAMS}
    return p, grad, m, v


ADAM_LR = dict(means=1.6e-4, log_scales=5e-3, quats=1e-3, opacity_logits=5e-2, sh=2.5e-3)
ADAM_STEP = 100


def prepare(case, seed):
    kind = case["kind"]
    s = SimpleNamespace(case=case, kind=kind)
    if kind == "adam":
        s.p, s.grad, s.m, s.v = _adam_inputs(case, seed)
        return s
    if kind == "densify":
        s.inputs = _densify_inputs(case, seed)
        return s
    s.hw = np.array([(h, w) for w, h in _sizes(case["views"])], np.int32)
    if kind in ("loss", "loss3d"):
        s.img, s.tgt = _image_pair(case["views"], seed)
        s.loss, s.dimg = torch.empty(len(s.hw), device="cuda"), torch.empty_like(s.img)
        if kind == "loss":
            s.ws = torch.empty(mvgs.dssim_workspace_size(s.hw), dtype=torch.uint8, device="cuda")
        else:
            s.pts, s.sig = _surface(case["views"], seed)
            s.ws = torch.empty(mvgs.dssim3d_workspace_size(s.hw), dtype=torch.uint8, device="cuda")
        return s
    s.p = _scene(case["n"], case["sh"], seed)
    s.cams = _cameras(case["views"], case["radius"], seed)
    tile = tuple(int(x) for x in case["tile"].split("x"))
    s.rz = mvgs.Rasterizer(s.cams, tile=tile, smem_batch=case["batch"])
    s.sc = mvgs.make_scene(s.p, case["sh"])
    s.rz.reserve_for(s.sc)
    if kind == "render":
        return s
    s.tgt = _targets(case["views"], seed)
    if kind == "autograd":
        for t in s.p.values():
            t.requires_grad_(True)
        return s
    s.grads = {k: torch.empty_like(t) for k, t in s.p.items()}
    s.dimg = torch.empty_like(s.tgt)
    if kind == "train":
        s.loss = torch.empty(s.cams.V, device="cuda")
        s.ws = torch.empty(mvgs.dssim_workspace_size(s.hw), dtype=torch.uint8, device="cuda")
    else:
        s.seed = int(seed)
        s.mhw = s.hw[:1]
        s.ws = torch.empty(mvgs.dssim3d_workspace_size(s.mhw), dtype=torch.uint8, device="cuda")
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _backward_and_statistics(s, samples=None):
    n, R = s.case["n"], max(int(s.rz.needed.records), 1)
    gm2d, e1 = torch.empty(R, 2, device="cuda"), torch.empty(R, device="cuda")
    s.rz.backward(s.sc, s.dimg, s.grads, gm2d, e1, samples=samples)
    acc = [torch.zeros(n, device="cuda") for _ in range(3)]
    mvgs.adc_accumulate(s.rz.state, n, gm2d, e1, *acc)
    return acc


def run(s):
    kind = s.kind
    if kind == "autograd":
        for t in s.p.values():
            t.grad = None
        img = autograd.render(s.rz, s.p, s.case["sh"])
        loss = (img - s.tgt).abs().mean()
        loss.backward()
        return dict(img=img.detach(), loss=loss.detach(), grads={k: s.p[k].grad for k in PARAMS})
    if kind == "train":
        img = s.rz.forward(s.sc)
        mvgs.dssim_loss(img, s.tgt, s.hw, LAMBDA, s.loss, s.dimg, s.ws)
        acc = _backward_and_statistics(s)
        return dict(img=img, loss=s.loss, grads=s.grads, acc=acc)
    if kind == "partial":
        c, V, rz = s.rz.cams_c, s.cams.V, s.rz
        P = int(s.mhw[0, 0]) * int(s.mhw[0, 1])
        samples = rz.sample_set(V, s.seed)
        img = torch.zeros(3 * rz.pixels, device="cuda")
        rz.forward(s.sc, images=img, samples=samples, depth=True)
        rec = rz.records()
        mimg, mtgt, pts, dm = (torch.empty(3 * P, device="cuda") for _ in range(4))
        sig, loss = torch.empty(P, device="cuda"), torch.empty(1, device="cuda")
        mvgs.merge_views(c, V, s.seed, img, s.tgt, rec["depth_acc"], rec["final_T"], mimg, mtgt, pts, sig)
        mvgs.dssim3d_loss(mimg, mtgt, pts, sig, s.mhw, LAMBDA, loss, dm, s.ws)
        mvgs.split_merged_grad(c, V, s.seed, dm, s.dimg)
        acc = _backward_and_statistics(s, samples)
        return dict(img=img, points=pts, sigma=sig, loss=loss, dimg=s.dimg, grads=s.grads, acc=acc)
    if kind == "render":
        s.rz.set_cameras(s.cams)
        return s.rz.forward(s.sc)
    if kind == "loss":
        mvgs.dssim_loss(s.img, s.tgt, s.hw, LAMBDA, s.loss, s.dimg, s.ws)
        return dict(loss=s.loss, dimg=s.dimg)
    if kind == "loss3d":
        mvgs.dssim3d_loss(s.img, s.tgt, s.pts, s.sig, s.hw, LAMBDA, s.loss, s.dimg, s.ws)
        return dict(loss=s.loss, dimg=s.dimg)
    if kind == "adam":
        for k in PARAMS:
            mvgs.adam_step(s.p[k], s.grad[k], s.m[k], s.v[k], ADAM_LR[k], ADAM_STEP)
        return dict(p=s.p, m=s.m, v=s.v)
    p, e1, e2, denom, normals, carry, thr = s.inputs
    new, src, kinds, moved = mvgs.densify(p, s.case["sh"], e1, e2, denom, normals, *thr, carry=carry)
    return dict(new=new, src=src, kind=kinds, moved=moved)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    """Inputs read once, outputs written once; operations of a render from the
    (pixel, Gaussian) pairs Eq. 1 blends -- about 107 a pixel at 500k Gaussians
    and 190 at 3M, as the library's own pixel statistics count them -- at 22
    FLOP forward and 64 backward."""
    kind = case["kind"]
    if kind in ("loss", "loss3d"):
        P = _pixels(case["views"])
        if kind == "loss":  # two separable 11-tap blurs: 5 moments forward, 3 partials backward
            return dict(bytes=36.0 * P, flops=3.0 * P * 2 * 2 * 11 * 8)
        return dict(bytes=52.0 * P, flops=121.0 * P * (2 * 10 + 15 * 2 + 9 * 2))
    nk = 3 * (case["sh"] + 1) ** 2
    per = 4.0 * (11 + nk)  # bytes of one Gaussian's parameters
    n = case["n"]
    if kind == "adam":
        return dict(bytes=7.0 * per * n, flops=15.0 * per / 4 * n)
    if kind == "densify":  # about as many out as in, with both moments
        return dict(bytes=n * (6 * per + 36.0 + 12.0), flops=60.0 * n)
    P = _pixels(case["views"])
    blended = (P / len(_sizes(case["views"])) if kind == "partial" else P) * 107.0 * (n / 5e5) ** 0.32
    if kind == "render":
        return dict(bytes=per * n + 12.0 * P, flops=22.0 * blended)
    stats = 0.0 if kind == "autograd" else 12.0 * n
    return dict(bytes=2 * per * n + 24.0 * P + stats, flops=86.0 * blended)


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------
def exact(case, seed):
    kind = case["kind"]
    if kind == "adam":
        return _exact_adam(case, seed)
    if kind == "densify":
        return _exact_densify(case, seed)
    if kind == "loss":
        img, tgt = _image_pair(case["views"], seed)
        loss, dimg = _exact_dssim(img.double(), tgt.double(), _sizes(case["views"]))
        return dict(loss=loss, dimg=dimg)
    if kind == "loss3d":
        return _exact_dssim3d(case, seed)
    if kind == "partial" or case["n"] * _pixels(case["views"]) > 4e9:
        return None
    return _exact_render(case, seed)


def _exact_adam(case, seed):
    p, grad, m, v = _adam_inputs(case, seed)
    out = dict(p={}, m={}, v={})
    f32 = lambda x: float(np.float32(x))  # noqa: E731
    b1, b2, eps = f32(0.9), f32(0.999), f32(1e-15)
    for k in PARAMS:
        g = grad[k].double()
        mm = b1 * m[k].double() + (1 - b1) * g
        vv = b2 * v[k].double() + (1 - b2) * g * g
        step = f32(ADAM_LR[k]) * (mm / (1 - b1 ** ADAM_STEP)) / ((vv / (1 - b2 ** ADAM_STEP)).sqrt() + eps)
        out["p"][k], out["m"][k], out["v"][k] = p[k].double() - step, mm, vv
    return out


def _rotation(q):
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)


def _exact_densify(case, seed):
    p, e1, e2, denom, normals, carry, (t1, t2, prune, extent) = _densify_inputs(case, seed)
    d = {k: v.double() for k, v in p.items()}
    den = denom.double()
    mean = [torch.where(den > 0, e.double() / den, torch.zeros_like(den)) for e in (e1, e2)]
    large = d["log_scales"].max(dim=1).values > extent
    keep = ~(d["opacity_logits"] < prune)
    split = keep & large & (mean[0] >= t1)
    clone = keep & ~large & (mean[1] >= t2)
    count = keep.long() + (split | clone).long()
    src = torch.repeat_interleave(torch.arange(case["n"], device="cuda"), count)
    first = torch.cumsum(count, 0) - count
    k = torch.arange(src.numel(), device="cuda") - first[src]
    sp = split[src]
    new = {name: t[src] for name, t in d.items()}
    z = normals.double()[src, k]
    off = torch.einsum("nij,nj->ni", _rotation(d["quats"][src]), d["log_scales"][src].exp() * z)
    new["means"] = torch.where(sp[:, None], new["means"] + off, new["means"])
    new["log_scales"] = torch.where(sp[:, None], new["log_scales"] - math.log(1.6), new["log_scales"])
    kinds = torch.where(sp, torch.full_like(k, 2), k).int()
    moved = []
    for t in carry:
        same = (kinds == 0).view(-1, *[1] * (t.dim() - 1))
        moved.append(torch.where(same, t.double()[src], torch.zeros((), dtype=torch.float64, device="cuda")))
    return dict(new=new, src=src, kind=kinds, moved=moved)


def _taps():
    x = torch.arange(-5, 6, dtype=torch.float64)
    w = torch.exp(-x * x / 4.5)
    return (w / w.sum()).tolist()


def _blur(x):
    w = _taps()
    h, wd = x.shape[-2:]
    x = torch.nn.functional.pad(x, (5, 5, 5, 5))
    x = sum(w[k] * x[..., k:k + wd] for k in range(11))
    return sum(w[k] * x[..., k:k + h, :] for k in range(11))


def _ssim(m1, m2, m11, m22, m12):
    c1, c2 = 0.01 ** 2, 0.03 ** 2
    t11, t22, t12 = m11 - m1 * m1, m22 - m2 * m2, m12 - m1 * m2
    return (2 * m1 * m2 + c1) * (2 * t12 + c2) / ((m1 * m1 + m2 * m2 + c1) * (t11 + t22 + c2))


def _exact_dssim(img, tgt, sizes):
    losses, grads, at = [], [], 0
    for w, h in sizes:
        a = img[at:at + 3 * w * h].view(3, h, w).clone().requires_grad_(True)
        b = tgt[at:at + 3 * w * h].view(3, h, w)
        at += 3 * w * h
        s = _ssim(_blur(a), _blur(b), _blur(a * a), _blur(b * b), _blur(a * b))
        loss = (1 - LAMBDA) * (a - b).abs().mean() + LAMBDA * (1 - s.mean())
        grads.append(torch.autograd.grad(loss / len(sizes), a)[0].reshape(-1))
        losses.append(loss.detach())
    return torch.stack(losses), torch.cat(grads)


def _exact_dssim3d(case, seed):
    img, tgt = _image_pair(case["views"], seed)
    pts, sig = _surface(case["views"], seed)
    (w, h), = _sizes(case["views"])
    a = img.double().view(3, h, w).requires_grad_(True)
    b, X, s = tgt.double().view(3, h, w), pts.double().view(3, h, w), sig.double().view(h, w)
    pad = lambda t: torch.nn.functional.pad(t, (5, 5, 5, 5))  # noqa: E731
    pa, pb, pX, ps = pad(a), pad(b), pad(X), pad(s)
    Z, sums = 0.0, [0.0] * 5
    for dv in range(11):
        for du in range(11):
            cut = lambda t: t[..., dv:dv + h, du:du + w]  # noqa: E731
            if du == 5 and dv == 5:
                k = torch.ones_like(s)
            else:
                ok = (s > 0) & (cut(ps) > 0)
                k = torch.where(ok, torch.exp(-((cut(pX) - X) ** 2).sum(0) / torch.where(ok, 2 * s * s, 1.0)), 0.0)
            Z = Z + k
            u, v = cut(pa), cut(pb)
            for i, t in enumerate((u, v, u * u, v * v, u * v)):
                sums[i] = sums[i] + k * t
    loss = (1 - LAMBDA) * (a - b).abs().mean() + LAMBDA * (1 - _ssim(*[t / Z for t in sums]).mean())
    return dict(loss=loss.detach().reshape(1), dimg=torch.autograd.grad(loss, a)[0].reshape(-1))


def _sh_basis(d, deg):
    x, y, z = d.unbind(1)
    pi = math.pi
    b = [torch.full_like(x, 0.5 * math.sqrt(1 / pi))]
    if deg > 0:
        c = math.sqrt(3 / (4 * pi))
        b += [-c * y, c * z, -c * x]
    if deg > 1:
        c, c0, c2 = 0.5 * math.sqrt(15 / pi), 0.25 * math.sqrt(5 / pi), 0.25 * math.sqrt(15 / pi)
        b += [c * x * y, -c * y * z, c0 * (2 * z * z - x * x - y * y), -c * x * z, c2 * (x * x - y * y)]
    if deg > 2:
        a, bb, c = 0.25 * math.sqrt(35 / (2 * pi)), 0.5 * math.sqrt(105 / pi), 0.25 * math.sqrt(21 / (2 * pi))
        d0, e = 0.25 * math.sqrt(7 / pi), 0.25 * math.sqrt(105 / pi)
        xx, yy, zz = x * x, y * y, z * z
        b += [-a * y * (3 * xx - yy), bb * x * y * z, -c * y * (4 * zz - xx - yy), d0 * z * (2 * zz - 3 * xx - 3 * yy),
              -c * x * (4 * zz - xx - yy), e * z * (xx - yy), -a * x * (xx - 3 * yy)]
    return torch.stack(b, 1)


def _project(p, cam, v, tile, deg):
    """The visible Gaussians of one view, by depth: indices and (xy, conic, opacity, rgb, radius)."""
    f64 = dict(dtype=torch.float64, device="cuda")
    vm = torch.tensor(cam.viewmat[v], **f64)
    fx, fy, cx, cy = (float(getattr(cam, k)[v]) for k in ("fx", "fy", "cx", "cy"))
    W, H = int(cam.width[v]), int(cam.height[v])
    R = vm[:, :3]
    t = p["means"] @ R.T + vm[:, 3]
    seen = t[:, 2] > float(cam.near[v])
    tz = torch.where(seen, t[:, 2], torch.ones_like(t[:, 2]))
    ux, uy = t[:, 0] / tz, t[:, 1] / tz
    lx, ly = 1.3 * 0.5 * W / fx, 1.3 * 0.5 * H / fy
    zero = torch.zeros_like(ux)
    J = torch.stack([fx / tz, zero, -fx * ux.clamp(-lx, lx) / tz, zero, fy / tz, -fy * uy.clamp(-ly, ly) / tz], 1)
    M = _rotation(p["quats"]) * p["log_scales"].exp()[:, None, :]
    TM = (J.view(-1, 2, 3) @ R) @ M
    S = TM @ TM.transpose(1, 2)
    a, b, c = S[:, 0, 0] + 0.3, S[:, 0, 1], S[:, 1, 1] + 0.3
    det = a * c - b * b
    xy = torch.stack([fx * ux + cx, fy * uy + cy], 1)
    o = torch.sigmoid(p["opacity_logits"])
    with torch.no_grad():
        mid = 0.5 * (a + c)
        r = torch.ceil(3 * torch.sqrt(mid + torch.sqrt((mid * mid - det).clamp(min=0.1))))
        lo = torch.log(255 * o)
        ext = 2 * lo.clamp(min=0) * 1.001 + 1e-3
        seen = seen & (det > 0) & (lo > 0)
        for q, sd, step, size in ((xy[:, 0], a, tile[0], W), (xy[:, 1], c, tile[1], H)):
            half = torch.minimum(r, torch.sqrt(ext * sd) + 1e-2)
            tiles = -(-size // step)
            seen = seen & (torch.floor((q - half) / step).clamp(0, tiles) <
                           (torch.floor((q + half) / step) + 1).clamp(0, tiles))
        ids = seen.nonzero()[:, 0]
        ids = ids[torch.sort(t[ids, 2].float(), stable=True).indices]
    d = p["means"] - torch.tensor(cam.campos[v], **f64)
    Y = _sh_basis(d / d.norm(dim=1, keepdim=True), deg)
    rgb = (torch.einsum("nk,nkc->nc", Y, p["sh"]) + 0.5).clamp(min=0)
    conic = torch.stack([c / det, -b / det, a / det], 1)
    return ids, xy[ids], conic[ids], o[ids], rgb[ids], r[ids]


def _pairs(px, py, xy, conic, o, r):
    dx, dy = px[:, None] - xy[None, :, 0], py[:, None] - xy[None, :, 1]
    A, B, C = conic[None].unbind(2)
    power = -0.5 * (A * dx * dx + C * dy * dy) - B * dx * dy
    G = torch.exp(power)
    raw = o[None] * G
    alpha = raw.clamp(max=0.99)
    ok = (dx.abs() <= r[None]) & (dy.abs() <= r[None]) & (power <= 0) & (alpha >= 1 / 255)
    alpha = torch.where(ok, alpha, 0.0)
    stopped = torch.cumprod(1 - alpha, 1) < 1e-4
    alpha = torch.where(torch.cumsum(stopped, 1) > 0, 0.0, alpha)
    after = torch.cumprod(1 - alpha, 1)
    T = torch.cat([torch.ones_like(after[:, :1]), after[:, :-1]], 1)
    return dx, dy, G, alpha, raw < 0.99, T, after[:, -1]


def _exact_render(case, seed):
    deg, tile = case["sh"], tuple(int(x) for x in case["tile"].split("x"))
    p = {k: v.double().requires_grad_(True) for k, v in _scene(case["n"], deg, seed).items()}
    cam = _cameras(case["views"], case["radius"], seed)
    sizes = _sizes(case["views"])
    recs, imgs = [], []
    for v, (w, h) in enumerate(sizes):
        ids, *rec = _project(p, cam, v, tile, deg)
        recs.append((ids, rec))
        xy, conic, o, rgb, r = (t.detach() for t in rec)
        out = torch.zeros(3, h * w, dtype=torch.float64, device="cuda")
        for pix in torch.arange(h * w, device="cuda").split(max(1, 20_000_000 // max(1, ids.numel()))):
            if ids.numel():
                _, _, _, alpha, _, T, _ = _pairs(pix % w + 0.5, pix // w + 0.5, xy, conic, o, r)
                out[:, pix] = ((alpha * T) @ rgb).T
        imgs.append(out.reshape(-1))
    img = torch.cat(imgs)
    if case["kind"] == "render":
        return img
    tgt = _targets(case["views"], seed).double()
    if case["kind"] == "autograd":
        loss, dimg = (img - tgt).abs().mean(), torch.sign(img - tgt) / img.numel()
    else:
        loss, dimg = _exact_dssim(img, tgt, sizes)
    n, at = case["n"], 0
    acc = [torch.zeros(n, dtype=torch.float64, device="cuda") for _ in range(3)]
    for (ids, rec), (w, h) in zip(recs, sizes):
        d_img = dimg[at:at + 3 * w * h].view(3, h * w)
        at += 3 * w * h
        if not ids.numel():
            continue
        xy, conic, o, rgb, r = (t.detach() for t in rec)
        g = [torch.zeros_like(t) for t in (xy, conic, o, rgb)]
        e1 = torch.zeros_like(o)
        A, B, C = conic[None].unbind(2)
        for pix in torch.arange(h * w, device="cuda").split(max(1, 20_000_000 // ids.numel())):
            dx, dy, G, alpha, free, T, _ = _pairs(pix % w + 0.5, pix // w + 0.5, xy, conic, o, r)
            d = d_img[:, pix].T
            dc = d @ rgb.T
            part = alpha * T * dc
            behind = part.sum(1, keepdim=True) - torch.cumsum(part, 1)
            da = torch.where((alpha > 0) & free, T * dc - behind / (1 - alpha), 0.0)
            dp = da * alpha
            ax, ay = A * dx + B * dy, B * dx + C * dy
            g[0] += torch.stack([(dp * ax).sum(0), (dp * ay).sum(0)], 1)
            g[1] += torch.stack([-0.5 * (dp * dx * dx).sum(0), -(dp * dx * dy).sum(0), -0.5 * (dp * dy * dy).sum(0)], 1)
            g[2] += (da * G).sum(0)
            g[3] += (alpha * T).T @ d
            e1 += (dp.abs() * torch.sqrt(ax * ax + ay * ay)).sum(0)
        torch.autograd.backward(rec[:4], g)
        acc[0][ids] += e1
        acc[1][ids] += g[0].norm(dim=1)
        acc[2][ids] += 1
    grads = {k: p[k].grad if p[k].grad is not None else torch.zeros_like(p[k]) for k in PARAMS}
    out = dict(img=img, loss=loss, grads=grads)
    return out if case["kind"] == "autograd" else dict(out, acc=acc)
