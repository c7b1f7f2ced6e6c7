"""The 3D D-SSIM's packed loops and its general ones: a value that sends a block to
the general loops changes nothing beyond the pixels it reaches, bit for bit, and
image sizes around the two-row lanes and the 32 x 8 blocks match the oracle."""
import numpy as np
import pytest
import torch

from gpu_helpers import assert_close_frac
from oracle import dssim3d

pytestmark = pytest.mark.gpu


def _inputs(W, H, seed):
    rng = np.random.default_rng(seed)
    cam = dict(W=W, H=H, fx=60.0, fy=60.0, cx=W / 2, cy=H / 2, R=np.eye(3), t=np.zeros(3))
    depth = 2.0 + 0.3 * rng.uniform(size=(H, W)) + np.linspace(0, 1, W)[None, :]
    T = np.where(rng.uniform(size=(H, W)) < 0.05, 1.0 - 1e-5, rng.uniform(0, 0.5, size=(H, W)))
    X, S = dssim3d.lift(depth * (1 - T), T, cam)
    a = rng.uniform(size=(3, H, W))
    b = np.clip(a + rng.normal(0, 0.2, size=a.shape), 0, 1)
    return [v.astype(np.float32) for v in (a, b, X, S)]


def _loss(mvgs, arrays, lam=0.2):
    H, W = arrays[0].shape[1:]
    hw = np.array([[H, W]], np.int32)
    t = [torch.tensor(v.reshape(-1), device="cuda") for v in arrays]
    ws = torch.empty(mvgs.dssim3d_workspace_size(hw), dtype=torch.uint8, device="cuda")
    loss, d = torch.empty(1, device="cuda"), torch.empty(3 * H * W, device="cuda")
    mvgs.dssim3d_loss(*t, hw, lam, loss, d, ws)
    return loss.item(), d.cpu().numpy().reshape(3, H, W)


@pytest.mark.parametrize("which,value", [(0, np.inf), (1, np.nan), (0, 1e30), (2, 2.0 ** 30), (2, np.nan), (2, np.inf),
                                         (3, 2.0 ** -30), (3, np.inf), (3, 1e-42), (3, np.nan), (3, -3.0)])
@pytest.mark.parametrize("at", [(40, 31), (47, 32), (33, 60)])
def test_an_odd_value_stays_within_two_windows(cuda_lib, which, value, at):
    W, H = 96, 80
    arrays = _inputs(W, H, 5)
    arrays[3][at] = 0.05
    _, clean = _loss(cuda_lib, arrays)
    arrays[which][(0, *at) if which < 3 else at] = value
    _, got = _loss(cuda_lib, arrays)
    y, x = np.mgrid[:H, :W]
    far = np.maximum(abs(y - at[0]), abs(x - at[1])) > 10
    np.testing.assert_array_equal(got[:, far], clean[:, far])


@pytest.mark.parametrize("W,H", [(1, 1), (40, 1), (33, 2), (31, 7), (32, 8), (65, 9), (5, 27)])
@pytest.mark.parametrize("lam", [0.2, 1.0])
def test_sizes_match_the_oracle(cuda_lib, W, H, lam):
    arrays = _inputs(W, H, W + 7 * H)
    L, g, _ = dssim3d.dssim3d_loss(*[v.astype(np.float64) for v in arrays], lam)
    loss, d = _loss(cuda_lib, arrays, lam)
    assert abs(loss - L) < 2e-6
    assert_close_frac(d, g, 1e-3, 1e-4 * np.abs(g).max(), "dL/dI")
