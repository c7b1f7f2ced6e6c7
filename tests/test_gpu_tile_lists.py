"""The per-tile lists built through bins of 8 x 8 tiles equal the oracle's
(view, tile, depth, Gaussian) sort of the same records, bit for bit: entry
counts around the chunks of 1024 entries and the groups of 32, rectangles that
cross bin edges, one bin (no sort pass), few bins (a narrow pass), more than
256 (two passes), and more than 2^20 (bin ids that leave no room for the local
rectangle in the sort key)."""
import numpy as np
import pytest

import oracle
import synth
from gpu_helpers import dense_records, gpu_forward

pytestmark = pytest.mark.gpu


def _check(cuda_lib, scene, cams, tile):
    rz, _, _, _ = gpu_forward(cuda_lib, scene, cams, tile)
    D = dense_records(rz, scene.n, cams.V)
    vis = D["valid"] != 0
    depth32 = np.zeros(scene.n * cams.V, np.float32)
    depth32[vis] = D["raw"]["depth"][D["rec_index"][vis]]
    keys, recs, ranges = oracle.sort_keys(cams, tile, D["valid"], D["rect"], depth32)
    got = D["raw"]["sorted"].astype(np.int64)
    np.testing.assert_array_equal(D["raw"]["v"][got].astype(np.int64) * scene.n + D["raw"]["g"][got], recs)
    gr = D["raw"]["ranges"]
    np.testing.assert_array_equal(gr[:, 1] - gr[:, 0], ranges[:, 1] - ranges[:, 0])
    some = ranges[:, 1] > ranges[:, 0]
    np.testing.assert_array_equal(gr[some], ranges[some])
    return rz


@pytest.mark.parametrize("n", [1, 31, 33, 1023, 1024, 1025, 2049])
@pytest.mark.parametrize("sizes,tile", [([(128, 128)], (16, 16)),       # one bin
                                        ([(129, 65)], (16, 16)),        # 9 x 5 tiles: two bins, the second one tile wide
                                        ([(640, 480)] * 3, (8, 8)),     # 240 bins: one full pass
                                        ([(72, 40)] * 150, (8, 8))])    # 300 bins: two passes, the second over one bit
def test_lists_equal_the_oracle_sort(cuda_lib, n, sizes, tile):
    if len(sizes) > 3 and n > 1025:
        n = 1025
    scene = synth.make_scene(n, 0, seed=n)
    scene.log_scales[:] -= np.float32(1.0)
    scene.log_scales[::7] += np.float32(2.5)  # some reach over many bins
    _check(cuda_lib, scene, synth.make_cameras(sizes, radius=3.0, seed=n + 1), tile)


def test_lists_with_more_bins_than_the_key_has_room_for(cuda_lib):
    V, H = 2050, 32760  # 512 bins per view: 1 x 4095 tiles
    n = 12
    rng = np.random.default_rng(5)
    scene = synth.make_scene(n, 0, seed=6)
    scene.means[:, 0] = 0.0
    scene.means[:, 1] = rng.uniform(-0.9, 0.9, n).astype(np.float32)
    scene.means[:, 2] = rng.uniform(1.9, 2.1, n).astype(np.float32)
    scene.log_scales[:] = np.float32(-5.5)
    scene.opacity_logits[:] = 1.0
    vm = np.zeros((V, 3, 4), np.float32)
    vm[:, :, :3] = np.eye(3, dtype=np.float32)
    f32 = np.float32
    cams = synth.Cameras(np.full(V, 1, np.int32), np.full(V, H, np.int32), np.full(V, 3e4, f32), np.full(V, 3e4, f32),
                         np.full(V, 0.5, f32), np.full(V, H / 2, f32), vm, np.zeros((V, 3), f32),
                         np.full(V, 0.2, f32))
    rz = _check(cuda_lib, scene, cams, (8, 8))
    assert int(rz.layout.tiles) == V * 4095 and int(rz.needed.keys) > V * n * 8


@pytest.mark.parametrize("tile", [(8, 8), (16, 8), (32, 32), (8, 64), (32, 64)])
def test_rectangles_for_any_tile(cuda_lib, tile):
    """A rectangle differs from the float64 one only where an edge falls on the rounding."""
    scene, cams = synth.make_scene(3000, 0, seed=2), synth.make_cameras([(301, 203), (97, 390)], radius=3.0, seed=3)
    rz, _, _, _ = gpu_forward(cuda_lib, scene, cams, tile)
    D, P = dense_records(rz, scene.n, cams.V), oracle.project(scene, cams, tile)
    vis = (D["valid"] != 0) & (P["valid"] != 0)
    assert vis.sum() > 2000
    assert (D["rect"][vis] != P["rect"][vis]).any(axis=1).mean() < 1e-3


def test_lists_sized_by_a_capacity_equal_the_exact_ones(cuda_lib):
    """A capturable render with room to spare, its launches striding over more radix
    blocks and chunks than they have blocks, against one sized by the counts."""
    scene = synth.make_scene(1_400_000, 0, seed=6)
    cams = synth.make_cameras([(1264, 832)] * 4, radius=4.0, seed=7)
    rz, sc, _, img = gpu_forward(cuda_lib, scene, cams, (16, 16))
    exact = rz.records()
    keys, records = exact["sorted"].shape[0], exact["g"].shape[0]
    assert keys > 4864 * 4096 * 14  # about 15 tiles per entry: more than 4864 radix blocks of 4096, and chunks by far
    cap = cuda_lib.Rasterizer(cams, tile=(16, 16), capturable=True)
    cap.reserve(scene.n, 6_000_000, keys + keys // 4)
    got = cap.forward(sc)
    assert bool((got == img).all())
    lists = cap.records()
    assert bool((lists["ranges"] == exact["ranges"]).all())
    assert bool((lists["sorted"][:keys] == exact["sorted"]).all())
    assert records <= 6_000_000
