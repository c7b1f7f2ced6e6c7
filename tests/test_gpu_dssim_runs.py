"""The l1 + D-SSIM loss over blocks that take runs of several tiles: a batch large
enough for them against its views one by one (a block per tile), bit for bit --
the batch's gradient is the view's divided by the number of views, a power of
two -- for heights around the 32-row tiles and the 10 rows that runs carry on."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _loss(mvgs, img, tgt, hw, lam):
    hw = np.array(hw, np.int32)
    ws = torch.empty(mvgs.dssim_workspace_size(hw), dtype=torch.uint8, device="cuda")
    loss, d = torch.empty(len(hw), device="cuda"), torch.full_like(img, float("nan"))
    mvgs.dssim_loss(img, tgt, hw, lam, loss, d, ws)
    return loss, d


@pytest.mark.parametrize("lam", [0.2, 1.0])
@pytest.mark.parametrize("sizes", [[(720, 330)] * 8, [(673, 500), (704, 31), (1, 700), (650, 650), (31, 64), (33, 33),
                                                      (736, 500), (1000, 1001)] * 2])
def test_runs_do_not_change_a_bit(cuda_lib, sizes, lam):
    g = torch.Generator("cuda").manual_seed(len(sizes))
    total = sum(3 * h * w for h, w in sizes)
    img = torch.rand(total, device="cuda", generator=g)
    tgt = (img + 0.2 * torch.randn(total, device="cuda", generator=g)).clamp(0, 1)
    loss, d = _loss(cuda_lib, img, tgt, sizes, lam)
    at = 0
    for v, (h, w) in enumerate(sizes):
        part = slice(at, at + 3 * h * w)
        at += 3 * h * w
        one_loss, one = _loss(cuda_lib, img[part].clone(), tgt[part].clone(), [(h, w)], lam)
        assert torch.equal(loss[v], one_loss[0])
        assert torch.equal(d[part] * len(sizes), one)
