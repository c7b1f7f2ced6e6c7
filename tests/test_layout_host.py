"""Buffer sizes on the host: state and workspace together hold no more per record and
key than 100 and 21 bytes (about what they took before the blend's 32-byte geometry
records), from three keys per record on: a memory budget that held a batch still
does."""
import pytest

import synth


@pytest.fixture(scope="module")
def mvgs():
    from paper_2506_12727_gb300 import build
    build.build()
    from paper_2506_12727_gb300 import mvgs
    return mvgs


@pytest.mark.parametrize("n,R,K", [(3_000_000, 22_000_000, 340_000_000), (500_000, 2_000_000, 116_000_000),
                                   (2_000_000, 8_000_000, 24_000_000), (1_000_000, 5_000_000, 15_000_000),
                                   (200_000, 100_000, 1_000_000)])
@pytest.mark.parametrize("V,size,tile", [(8, (1264, 832), (32, 64)), (5, (1600, 1200), (16, 16)), (1, (640, 480), (8, 8))])
def test_state_and_workspace_stay_within_their_budget(mvgs, n, R, K, V, size, tile):
    cams = mvgs.make_cameras(synth.make_cameras([size] * V, radius=3.0, seed=1))
    L = mvgs.render_layout(n, cams, mvgs.make_config(tile), mvgs.Capacity(R, K))
    pixels, tiles = V * size[0] * size[1], int(L.tiles)
    before = 100 * R + 21 * K + (12 + V) * n + 22 * pixels + 80 * tiles
    assert L.state_bytes + L.workspace_bytes <= before + 500_000
