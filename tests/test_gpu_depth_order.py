"""The depth sort against a stable argsort of the depths' bits, in one tile that
every Gaussian covers: depth ranges on both sides of the pass widths (equal
depths, a few bits, 8, 9, 16, 18, 24, 25, 27, 28 and 32 bits, depths of both
signs), and counts around its blocks of 4096 keys, the 64 blocks up to which the
scatter sums the histograms itself, and the 5 and 1024 blocks where the scans
change."""
import math

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def _camera(near):
    f32 = np.float32
    f = f32(8.0 / math.tan(math.radians(30.0)))
    vm = np.zeros((1, 3, 4), f32)
    vm[0, :, :3] = np.eye(3)
    one = np.ones(1, f32)
    return synth.Cameras(np.array([16], np.int32), np.array([16], np.int32), f * one, f * one, 8 * one, 8 * one, vm,
                         np.zeros((1, 3), f32), near * one)


def _order(mvgs, z, near=0.1):
    n = z.shape[0]
    params = dict(means=torch.zeros(n, 3, device="cuda"), log_scales=torch.empty(n, 3, device="cuda"),
                  quats=torch.tensor([1.0, 0.0, 0.0, 0.0], device="cuda").repeat(n, 1),
                  opacity_logits=torch.full((n,), -3.0, device="cuda"), sh=torch.zeros(n, 1, 3, device="cuda"))
    params["means"][:, 2] = z
    params["log_scales"].copy_(torch.log(2.0 * z.abs())[:, None].expand(n, 3))
    rz = mvgs.Rasterizer(_camera(near), tile=(16, 16))
    sc = mvgs.make_scene(params, 0)
    rz.forward(sc)
    rec = rz.records()
    assert rec["g"].shape[0] == n
    assert torch.equal(rec["depth"], z)
    return rec["sorted"].long()


def _expected(z):
    bits = z.view(torch.int32).long() & 0xFFFFFFFF
    return torch.sort(bits, stable=True).indices


def _depths(n, bits, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    low = 0x3E4CCCCD  # 0.2
    span = (1 << bits) - 1
    k = torch.randint(0, span + 1, (n,), device="cuda", generator=g) + low
    k[0], k[-1] = low + span, low
    return k.to(torch.int32).view(torch.float32)


@pytest.mark.parametrize("bits", [0, 1, 5, 8, 9, 10, 16, 18, 19, 24, 25, 27, 28, 29])
@pytest.mark.parametrize("n", [2, 4095, 4097, 70001])
def test_depth_ranges(cuda_lib, bits, n):
    z = _depths(n, bits, bits + n)
    assert torch.equal(_order(cuda_lib, z), _expected(z))


@pytest.mark.parametrize("n", [1, 5 * 4096, 5 * 4096 + 1, 64 * 4096, 64 * 4096 + 1, 1024 * 4096, 1024 * 4096 + 1])
@pytest.mark.parametrize("bits", [12, 26])
def test_counts(cuda_lib, n, bits):
    z = _depths(n, bits, n)
    assert torch.equal(_order(cuda_lib, z), _expected(z))


def test_depths_of_both_signs(cuda_lib):
    g = torch.Generator("cuda").manual_seed(4)
    z = torch.rand(9000, device="cuda", generator=g) * 4.0 + 1.0
    z[::3] *= -1.0
    assert torch.equal(_order(cuda_lib, z, near=-10.0), _expected(z))
