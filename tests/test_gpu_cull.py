"""The rasterisers' ellipse cull of 8 x 8 blocks, splat by splat: one needle at a time, so
that a pixel the cull drops cannot hide in a scene-wide tolerance.

A map of a single splat with attribute 1 is its alpha where that reaches alpha_min, else 0.
Tolerance: the oracle flags the pixels whose decision lies within the a-priori FP32 error of
the exponent (oracle_raster.c: 16 u kappa p of that splat at that pixel, u = 2^-24); everywhere
else the two must agree on which pixels the splat reaches. Where both do, the values differ by
at most twice that error relative to alpha itself (the exponent's error is alpha's relative one;
the factor covers the kernel's exponential, 2 ulps, and the oracle's rounded inputs)."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2405_05446_gb300 as G
from paper_2405_05446_gb300 import scenes as S

from gpu_util import ensure_lib, gpu_maps, oracle_maps, oracle_opts
from test_gpu_raster import _needles

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


@pytest.mark.parametrize("hw,count", [((37, 61), 60), ((96, 130), 60), ((608, 1024), 24), ((640, 1024), 24)])
def test_no_pixel_of_a_needle_is_dropped(hw, count):
    """Sizes with ragged blocks, and both sides of the load-ahead line (2432 tiles)."""
    H, W = hw
    sc, cam = _needles(H + W, count, 1, True, W, H)
    ro = G.raster_opts(pairs_per_gaussian=256)
    amin = oracle_opts(ro).alpha_min
    edge = seen = 0
    for i in range(count):
        one = S.Scene(*(np.ascontiguousarray(a[i:i + 1]) for a in (sc.mean, sc.scale, sc.quat, sc.opacity)),
                      np.ones((1, 1), np.float32))
        gm, _, st = gpu_maps(one, cam, ro)
        assert st["status"] == 0, st
        om, amb = oracle_maps(one, cam, ro)
        gm, om, ok = gm[0], om[0], amb == 0
        assert np.array_equal((gm != 0)[ok], (om != 0)[ok]), i
        both = ok & (om != 0)
        if not both.any():
            continue
        proj = O.project(one, cam, oracle_opts(ro))[0]
        p = np.log(np.maximum(one.opacity[0] / om[both], 1.0))  # the exponent, >= 0
        tol = 2.0 * (16.0 * U * proj[O.KAPPA] * p + 8.0 * U)
        assert np.all(np.abs(gm - om)[both] <= tol * om[both]), i
        seen += int(both.sum())
        edge += int((both & (om < 1.5 * amin)).sum())
    assert seen > 100 * count / 4 and edge > count / 4  # pixels next to the cut were looked at
