"""The rasterisers' 8 x 8 warp blocks with two pixels per lane: image sizes that end inside
a block or a tile, elongated splats that cross blocks diagonally (the block cull follows
the ellipse, not its box), every attribute width, against the FP64 oracle.

Tolerance: the a-priori FP32 model of the exponent that the oracle's ambiguity flags use
(oracle_raster.c): an error of 16 u kappa p at a pixel p deep in a splat whose Sigma2D has
condition number kappa, u = 2^-24, p <= ln(255) where the splat contributes. It is a relative
error of alpha, of T and so of every weight: twice it bounds a map in units of the largest
attribute, four times it (alpha, T, the exponent's own factor and the offset) a gradient.
For round splats this is below the 1e-5 and 1e-4 of the other parity tests, which then
apply."""
import numpy as np
import pytest
import torch

import oracle as O
from oracle import diff as D
import paper_2405_05446_gb300 as G
from paper_2405_05446_gb300 import scenes as S

from gpu_util import AMB_FRAC_MAX, MAP_TOL, ensure_lib, gpu_maps, oracle_maps, oracle_opts

pytestmark = pytest.mark.gpu

GRAD_TOL = 1e-4
SMOOTH = dict(alpha_min=float(np.float32(1e-10)), alpha_max=0.99, t_min=0.0)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def _needles(seed, n, channels, laplacian, w, h):
    """Splats 20 to 60 times as long as wide at all angles, and round ones."""
    sc = S.tiny_scene(seed, n=n, channels=channels)
    rng = np.random.default_rng(seed)
    scale = sc.scale.copy()
    long = rng.random(n) < 0.7
    scale[long] = (np.stack([rng.uniform(0.2, 0.6, n), rng.uniform(0.008, 0.012, n),
                             rng.uniform(0.008, 0.012, n)], 1)[long]).astype(np.float32)
    sc = S.Scene(sc.mean * np.float32(0.7), scale, sc.quat, sc.opacity, sc.grad)
    if laplacian:
        sc = S.with_laplacian_attribute(sc, seed)
    return sc, S.look_at_camera((0.3, 0.2, -3.0), (0.0, 0.0, 0.0), w, h)


def _alpha_error(sc, cam, opts):
    proj = O.project(sc, cam, opts)
    kappa = proj[proj[:, O.VALID] > 0, O.KAPPA].max()
    return 16.0 * 2.0 ** -24 * kappa * np.log(255.0)


@pytest.mark.parametrize("hw", [(5, 3), (8, 8), (9, 17), (12, 40), (40, 12), (37, 61), (96, 130)])
@pytest.mark.parametrize("channels,laplacian", [(1, False), (3, False), (4, False), (1, True), (2, True), (3, True)])
def test_maps_of_needles_match_oracle(hw, channels, laplacian):
    H, W = hw
    sc, cam = _needles(H * 100 + W, 300, channels, laplacian, W, H)
    ro = G.raster_opts(pairs_per_gaussian=64)
    gm, _, st = gpu_maps(sc, cam, ro)
    assert st["status"] == 0 and st["n_pairs"] > 0
    om, amb = oracle_maps(sc, cam, ro)
    ok = amb == 0
    assert (~ok).sum() <= max(8, AMB_FRAC_MAX * 10 * amb.size)  # few pixels sit on a decision
    tol = max(MAP_TOL * np.abs(om).max(), 2.0 * _alpha_error(sc, cam, oracle_opts(ro)) * np.abs(sc.grad).max())
    assert np.abs(gm - om)[..., ok].max() <= tol


@pytest.mark.parametrize("hw", [(608, 1024), (609, 1024)])
@pytest.mark.parametrize("channels,laplacian", [(1, False), (3, False), (3, True)])
def test_maps_on_both_sides_of_the_load_ahead_line(hw, channels, laplacian):
    """2432 tiles, the most that load ahead, and one row of tiles more; lists of 0 to 300."""
    test_maps_of_needles_match_oracle(hw, channels, laplacian)


@pytest.mark.parametrize("hw", [(7, 13), (24, 40), (45, 33)])
@pytest.mark.parametrize("channels,laplacian", [(1, False), (3, False), (4, False), (1, True), (3, True)])
def test_gradients_of_needles_match_oracle(hw, channels, laplacian):
    H, W = hw
    sc, cam = _needles(H + W, 40, channels, laplacian, W, H)
    mean = [0.5] * channels
    w = np.random.default_rng(3).standard_normal((channels, H, W))
    ro, so = G.raster_opts(pairs_per_gaussian=256, **SMOOTH), G.solver_opts(rtol=1e-7)
    g = G.gaussians_to_device(sc)
    ws = torch.empty(G.workspace_size(sc.n, channels, W, H, ro, so), dtype=torch.uint8, device="cuda")
    ws_adj = torch.empty(G.workspace_size(0, channels, W, H, None, so), dtype=torch.uint8, device="cuda")
    img = torch.empty((channels, H, W), device="cuda")
    G.render_view(g, cam, mean, img, ws, ro, so)
    assert G.sync_status(ws)["status"] == 0
    gr = G.render_view_backward(g, cam, torch.as_tensor(w, dtype=torch.float32).cuda(), ws, ws_adj, ro, so)
    assert G.sync_status(ws_adj)["status"] == 0
    ref = D.gradients(sc, cam, mean, O.RasterOpts(**SMOOTH), w)
    tol = max(GRAD_TOL, 4.0 * _alpha_error(sc, cam, O.RasterOpts(**SMOOTH)))
    for k in D.PARAMS:
        a, b = gr[k].cpu().numpy().astype(np.float64).reshape(ref[k].shape), ref[k]
        assert np.abs(a - b).max() <= tol * np.abs(b).max(), k
