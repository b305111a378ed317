"""The workspace's size: what the sorts publish and the backward's sums lie on arrays that are
not live at the same time, so no image of a tile or more needs more than separate regions of
the earlier sorts' histograms and of 24 bytes per Gaussian would."""
import pytest

import paper_2405_05446_gb300 as G
from paper_2405_05446_gb300 import build as B


@pytest.fixture(scope="module", autouse=True)
def _lib():
    B.build()


def _up(b):
    return (b + 255) // 256 * 256


def _separate(n, C, W, H, ppg):
    cap, up = n * ppg, _up
    per_splat = 2 * up(16 * n) + up(8 * n) + 6 * up(4 * n)  # projected, keys and indices, tile counts
    pairs = 4 * up(4 * cap)
    hist = up(1024 * (max(-(-n // 512), -(-cap // 2048)) + 1))
    rest = up(8 * (-(-n // 256) + 2)) + up(8 * C * W * H) + up(24 * n)
    return G.workspace_size(0, C, W, H, None, None) + per_splat + pairs + hist + rest


@pytest.mark.parametrize("n", [1, 31, 161, 2048, 2049, 5000, 100003, 1000000])
@pytest.mark.parametrize("wh", [(16, 16), (24, 20), (129, 97), (640, 480), (3840, 2160)])
def test_size_is_not_above_separate_regions(n, wh):
    for C in (1, 3, 4):
        for ppg in (1, 2, 5, 16, 32, 64, 256):
            got = G.workspace_size(n, C, *wh, G.raster_opts(pairs_per_gaussian=ppg), None)
            assert 0 < got <= _separate(n, C, *wh, ppg), (n, C, wh, ppg)
