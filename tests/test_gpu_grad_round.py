"""The quaternion's gradient of nearly round splats, where it is what remains of terms that
nearly cancel: a rotation of a sphere changes nothing. In the splat's own frame it is the
torque 2 G_ij (s_i^2 - s_j^2) of the moments, whose differences are formed before any product
(backward.cu); through d R and moments of the offsets the same sums came out 1e-5 off.

Tolerance: no term cancels in that form, so the error (relative, 2-norm over the scene) is the
roundings of one chain: about 20 operations a pixel, 6 levels of FP32 sums over a block (the
blocks add up in FP64) and as many in the projection's transposes: 32 u, u = 2^-24."""
import numpy as np
import pytest
import torch

import oracle as O
from oracle import diff as D
import paper_2405_05446_gb300 as G
from paper_2405_05446_gb300 import scenes as S

from gpu_util import ensure_lib

pytestmark = pytest.mark.gpu

TOL = 32.0 * 2.0 ** -24
SMOOTH = dict(alpha_min=float(np.float32(1e-10)), alpha_max=0.99, t_min=0.0)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


@pytest.mark.parametrize("hw", [(96, 128), (255, 321)])
@pytest.mark.parametrize("seed", [0, 1, 2, 3])
def test_quaternion_gradient_of_nearly_round_splats(hw, seed):
    H, W = hw
    rng, n = np.random.default_rng(seed), 24
    sc = S.tiny_scene(seed, n=n, channels=1)
    q = rng.standard_normal((n, 4))
    size = rng.uniform(0.15, 0.3, n)
    scale = np.stack([size, size / 1.02, size / 1.02], 1).astype(np.float32)
    sc = S.Scene(sc.mean * np.float32(0.7), scale, (q / np.linalg.norm(q, axis=1, keepdims=True)).astype(np.float32),
                 np.full(n, 0.3, np.float32), sc.grad)
    cam = S.look_at_camera((0.3, 0.2, -3.0), (0.0, 0.0, 0.0), W, H)
    y, x = np.mgrid[0:H, 0:W]
    w = np.sin(6.0 * x / W + seed)[None] * np.cos(5.0 * y / H)
    mean = [0.5]
    ro, so = G.raster_opts(pairs_per_gaussian=512, **SMOOTH), G.solver_opts(rtol=1e-7)
    g = G.gaussians_to_device(sc)
    ws = torch.empty(G.workspace_size(n, 1, W, H, ro, so), dtype=torch.uint8, device="cuda")
    ws_adj = torch.empty(G.workspace_size(0, 1, W, H, None, so), dtype=torch.uint8, device="cuda")
    img = torch.empty((1, H, W), device="cuda")
    G.render_view(g, cam, mean, img, ws, ro, so)
    assert G.sync_status(ws)["status"] == 0
    gr = G.render_view_backward(g, cam, torch.as_tensor(w, dtype=torch.float32).cuda(), ws, ws_adj, ro, so)
    assert G.sync_status(ws_adj)["status"] == 0
    ref = D.gradients(sc, cam, mean, O.RasterOpts(**SMOOTH), w)
    for k in ("quat", "scale", "mean"):
        a = gr[k].cpu().numpy().astype(np.float64).reshape(ref[k].shape)
        assert np.linalg.norm(a - ref[k]) <= TOL * np.linalg.norm(ref[k]), k
