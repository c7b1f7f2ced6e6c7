"""The benchmark's byte counts of the stages that build the tile lists are those of
the kernels that build them: a fraction of the copy rate from them can be reached,
not passed."""
import os
import sys
import types

import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


def _records(rects, depths):
    return dict(rect=torch.tensor(rects, dtype=torch.int16), depth=torch.tensor(depths, dtype=torch.float32))


def test_list_work_counts_what_the_kernels_move():
    # rectangles of 1, 2 (across a bin edge), 4 (around a bin corner) and 9 bins, in tiles
    rects = [[0, 0, 8, 8], [7, 0, 9, 1], [7, 7, 9, 9], [4, 4, 20, 20]]
    K = 64 + 2 + 4 + 256
    rz = types.SimpleNamespace(n=4, layout=types.SimpleNamespace(tiles=40 * 30),
                               cfg=types.SimpleNamespace(tile_w=16, tile_h=16),
                               cams_np=types.SimpleNamespace(width=[640], height=[480]),
                               records=lambda: _records(rects, [2.0, 2.5, 3.0, 3.75]))
    w = bench.list_work(rz, (4, K))
    S, R = 1 + 2 + 4 + 9, 4
    # depths within a factor of two differ in 23 bits: three passes; 5 x 4 bins: one pass
    assert w["depth_sort"] == ("hbm", 60.0 * R, "B")
    assert w["tile_sort"] == ("hbm", 16.0 * R + 44.0 * S + 4.0 * K, "B")
    assert w["ranges"] == ("hbm", 72.0 * 1200, "B")
    # far fewer bytes than the sort of all (record, tile) pairs that came before
    before, _ = bench.stage_work(rz, (4, K), 1, 640 * 480, 1)
    assert w["tile_sort"][1] < 0.4 * before["tile_sort"][1]


def test_one_depth_and_one_bin_take_no_more_passes_than_they_need():
    rz = types.SimpleNamespace(n=1, layout=types.SimpleNamespace(tiles=4), cfg=types.SimpleNamespace(tile_w=16, tile_h=16),
                               cams_np=types.SimpleNamespace(width=[32], height=[32]),
                               records=lambda: _records([[0, 0, 2, 2]], [2.0]))
    w = bench.list_work(rz, (1, 4))
    assert w["depth_sort"] == ("hbm", 20.0, "B")
    assert w["tile_sort"] == ("hbm", 16.0 + 24.0 + 16.0, "B")
