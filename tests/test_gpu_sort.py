"""Binning (csrc/sort.cu) at the sizes where its radix passes and the pair emission change:
one Gaussian, the edges of a warp, of a block of the emission (256), of a tile of the depth
sort (2048) and more than one group of 16 tiles of either sort; images of one tile, of 257
tiles (9-bit keys: two passes) and of one row of tiles; no pairs; more pairs than the buffer.

The maps are compared with the oracle, which composites in depth order: a pair lost, doubled
or out of order shows in them. Tolerance: that of the other map tests (MAP_TOL of the largest
value), at pixels that sit on no decision."""
import numpy as np
import pytest

import oracle as O
import paper_2405_05446_gb300 as G
from paper_2405_05446_gb300 import scenes as S

from gpu_util import AMB_FRAC_MAX, MAP_TOL, ensure_lib, gpu_maps, oracle_maps

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def _scene(n, w, h):
    """Small faint splats over the whole image, all of them in front of the camera."""
    rng = np.random.default_rng(n + w)
    cam = S.look_at_camera((0.0, 0.0, -3.0), (0.0, 0.0, 0.0), w, h)
    sc = S.tiny_scene(n, n=n, channels=1)
    half = 1.4 * max(w, h) / (2.0 * cam.fx)
    mean = np.stack([rng.uniform(-half, half, n) * 2, rng.uniform(-half, half, n) * 2 * min(1.0, h / w),
                     rng.uniform(-0.6, 0.6, n)], 1).astype(np.float32)
    scale = np.full((n, 3), 0.6 * 3.0 / cam.fx, np.float32) * rng.uniform(0.5, 2.0, (n, 1)).astype(np.float32)
    opacity = rng.uniform(0.05, 0.5, n).astype(np.float32)
    return S.Scene(mean, scale, sc.quat, opacity.reshape(sc.opacity.shape), sc.grad), cam


@pytest.mark.parametrize("wh", [(16, 16), (4112, 16), (130, 90)])
@pytest.mark.parametrize("n", [1, 32, 33, 256, 257, 2047, 2048, 2049, 48000])
def test_maps_match_oracle_at_sort_edges(n, wh):
    sc, cam = _scene(n, *wh)
    ro = G.raster_opts(pairs_per_gaussian=8)
    gm, _, st = gpu_maps(sc, cam, ro)
    assert st["status"] == 0
    om, amb = oracle_maps(sc, cam, ro)
    ok = amb == 0
    assert (~ok).sum() <= max(8, AMB_FRAC_MAX * 10 * amb.size)
    assert np.abs(gm - om)[..., ok].max() <= MAP_TOL * max(np.abs(om).max(), np.abs(sc.grad).max() * 1e-3)
    again, _, st2 = gpu_maps(sc, cam, ro)
    assert np.array_equal(gm, again) and st2["n_pairs"] == st["n_pairs"]
    if n == 48000 and wh != (16, 16):
        assert st["n_pairs"] > 16 * 2560


@pytest.mark.parametrize("n", [300, 5000])
def test_more_pairs_than_the_buffer_holds(n):
    sc, cam = _scene(n, 130, 90)
    sc = S.Scene(sc.mean, sc.scale * np.float32(8), sc.quat, sc.opacity, sc.grad)
    _, _, st = gpu_maps(sc, cam, G.raster_opts(pairs_per_gaussian=1))
    assert st["status"] == G._abi.ERR_CAPACITY and st["n_pairs"] > n


def test_no_pairs():
    sc, cam = _scene(3000, 130, 90)
    sc = S.Scene(sc.mean - np.float32([0, 0, 50]), sc.scale, sc.quat, sc.opacity, sc.grad)  # all behind
    gm, _, st = gpu_maps(sc, cam, G.raster_opts(pairs_per_gaussian=4))
    assert st["status"] == 0 and st["n_pairs"] == 0 and not gm.any()
