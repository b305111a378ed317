"""The later cycles of the direct solve (csrc/fct.cu): each correction is a part of its own,
so a third cycle takes the residual below what FP32 holds of the second.

Tolerance: as test_gpu_fct.py, 1e-5 of the image's range; smooth fields of large images are
the ones that need the cycles (their Laplacian is 1e-6 of them)."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2405_05446_gb300 as G

from gpu_util import ensure_lib

pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def _solve(rho, **opts):
    C, H, W = rho.shape
    so = G.solver_opts(**opts)
    ws = torch.empty(G.workspace_size(0, C, W, H, None, so), dtype=torch.uint8, device="cuda")
    img = torch.empty((C, H, W), device="cuda")
    G.poisson_reconstruct_rho(torch.as_tensor(rho).cuda(), [0.0] * C, img, ws, sopts=so)
    return img.cpu().numpy().astype(np.float64), G.sync_status(ws)


def _smooth(kind, H, W):
    y, x = np.mgrid[0:H, 0:W]
    y, x = (y + 0.5) / H, (x + 0.5) / W
    if kind == "mode":
        return np.cos(np.pi * x)
    if kind == "blob":
        return np.exp(-20.0 * ((x - 0.5) ** 2 + (y - 0.4) ** 2))
    return np.sin(5.0 * x) * np.cos(4.0 * y)


@pytest.mark.parametrize("hw", [(2160, 3840), (4096, 4096), (2153, 3833)])
@pytest.mark.parametrize("kind", ["mode", "blob", "sin"])
@pytest.mark.parametrize("rtol", [1e-7])
def test_smooth_fields_of_large_images_meet_a_tight_rtol(hw, kind, rtol):
    """1e-7 is what the multigrid cycles accepted here. The floor of three corrections is L of the
    FP32 rounding of the third one, which the lowest modes dominate: up to 3e-8 (lowest mode, 3833 x 2153)."""
    rho = _smooth(kind, *hw).astype(np.float32)[None]
    img, st = _solve(rho, rtol=rtol, max_cycles=30)
    assert st["status"] == 0 and st["rel_residual"] <= rtol and st["cycles"] <= 3, st
    f = rho.astype(np.float64)
    ref = O.poisson_neumann(f - f.mean(), [0.0])
    assert np.abs(img - ref).max() <= TOL * (ref.max() - ref.min())


@pytest.mark.parametrize("hw", [(96, 128), (97, 101), (270, 481), (757, 1355)])
def test_channels_that_stop_after_different_cycles(hw):
    """A smooth channel (three cycles), a noisy one and a zero one at rtol = 1e-9: each image is
    that of its own 1-channel solve (to the last bit of the mean's shift) and of the oracle."""
    H, W = hw
    rng = np.random.default_rng(H)
    rho = np.stack([_smooth("mode", H, W), rng.laplace(0, 0.05, (H, W)), np.zeros((H, W))]).astype(np.float32)
    img, st = _solve(rho, rtol=1e-9, max_cycles=30)
    assert st["status"] == 0 and st["cycles"] == 3 and st["rel_residual"] <= 1e-9, st
    f = rho.astype(np.float64)
    ref = O.poisson_neumann(f - f.mean(axis=(1, 2), keepdims=True), [0.0] * 3)
    for c, cycles in enumerate(((3,), (2, 3), (0,))):
        one, st1 = _solve(rho[c:c + 1], rtol=1e-9, max_cycles=30)
        assert st1["status"] == 0 and st1["cycles"] in cycles, (c, st1)
        scale = np.abs(one).max()
        assert np.abs(one[0] - img[c]).max() <= 2.0 ** -22 * scale
        assert np.abs(img[c] - ref[c]).max() <= TOL * scale


def test_two_cycles_are_as_with_more_allowed():
    """Where two cycles meet rtol, a third that may run changes nothing."""
    rng = np.random.default_rng(5)
    rho = rng.laplace(0, 0.05, (2, 120, 200)).astype(np.float32)
    a, sa = _solve(rho, max_cycles=2)
    b, sb = _solve(rho, max_cycles=30)
    assert sa["status"] == sb["status"] == 0 and sa["cycles"] == sb["cycles"] == 2
    assert np.abs(a - b).max() <= 2.0 ** -22 * np.abs(a).max()
