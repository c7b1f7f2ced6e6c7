"""3D D-SSIM on coordinates and widths far from 1: only quotients of both enter, so
scaling both by a power of two changes no bit, in the packed loops' domain
(coordinates up to 2^30) or out of it, and out of it costs no more than the tests
that the general loops make."""
import numpy as np
import pytest
import torch

from test_gpu_dssim3d_paths import _inputs, _loss

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("power", [-24, -12, 10, 25, 30, 45])  # the last two out of the domain
def test_scaled_scenes_give_the_same_bits(cuda_lib, power):
    arrays = _inputs(101, 43, 8)
    L, g = _loss(cuda_lib, arrays)
    scaled = arrays[:2] + [a * np.float32(2.0 ** power) for a in arrays[2:]]
    L2, g2 = _loss(cuda_lib, scaled)
    assert L2 == L and np.array_equal(g2, g)


def _ms(cuda_lib, arrays):
    best = float("inf")
    cuda_lib.profile_enable(True)
    try:
        for _ in range(6):
            cuda_lib.profile_read()
            _loss(cuda_lib, arrays)
            torch.cuda.synchronize()
            best = min(best, cuda_lib.profile_read()["dssim"][0])
    finally:
        cuda_lib.profile_enable(False)
    return best


def test_large_coordinates_take_no_longer(cuda_lib):
    """A scene in metres on a map (coordinates of 2^22) as long as one around the
    origin; with values that only the general loops take, less than three times that
    (5.7 times when they read their windows from memory)."""
    arrays = _inputs(1264, 832, 8)
    plain = _ms(cuda_lib, arrays)
    far = _ms(cuda_lib, arrays[:2] + [a * np.float32(2.0 ** 22) for a in arrays[2:]])
    odd = [a.copy() for a in arrays]
    odd[0][0, 3::8, 7::32] = np.nan  # a pixel in every block
    general = _ms(cuda_lib, odd)
    assert far < 1.25 * plain and general < 3.0 * plain, (plain, far, general)


def test_background_is_passed_over(cuda_lib):
    """Pixels without a surface point have no window: an image of them takes less
    than two thirds of the time (as much when every warp walked its windows)."""
    arrays = _inputs(1264, 832, 8)
    plain = _ms(cuda_lib, arrays)
    arrays[3][:] = 0.0
    background = _ms(cuda_lib, arrays)
    assert background < 0.67 * plain, (plain, background)
