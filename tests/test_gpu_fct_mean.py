"""The direct solve (csrc/fct.cu) on fields whose mean is large against their variation: a
Laplacian field whose sum is not zero is solved in the least-squares sense (the mean comes
off), and the adjoint of a loss against a brighter target is such a field.

Tolerance: as test_gpu_fct.py, 1e-5 of the image's range against the exact DCT solution of
the FP32 field itself. The residual reported is that of the iterate: the returned image is
the iterate rounded to FP32, so its own residual exceeds the reported one by at most L of
that rounding, 8 half ulps of its largest value per pixel."""
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


def _laplacian(u):
    p = np.pad(u, 1, mode="edge")
    return p[1:-1, 2:] + p[1:-1, :-2] + p[2:, 1:-1] + p[:-2, 1:-1] - 4.0 * u


def _solve(rho, mean, **opts):
    """rho: FP32 [H][W]; the image in FP64 and the statistics."""
    H, W = rho.shape
    so = G.solver_opts(**opts)
    ws = torch.empty(G.workspace_size(0, 1, W, H, None, so), dtype=torch.uint8, device="cuda")
    img = torch.empty((1, H, W), device="cuda")
    G.poisson_reconstruct_rho(torch.as_tensor(rho[None]).cuda(), [mean], img, ws, sopts=so)
    return img[0].cpu().numpy().astype(np.float64), G.sync_status(ws)


def _noisy(H, W, seed):
    rng = np.random.default_rng(seed)
    y, x = np.mgrid[0:H, 0:W]
    return 0.5 + 0.3 * np.sin(5.0 * x / W) * np.cos(4.0 * y / H) + 0.02 * rng.standard_normal((H, W))


@pytest.mark.parametrize("hw", [(120, 200), (97, 101), (757, 1355), (1080, 1920)])
@pytest.mark.parametrize("ratio", [0.0, 3.0, 30.0, 300.0, -3000.0])
def test_field_with_a_large_mean(hw, ratio):
    H, W = hw
    lap = _laplacian(_noisy(H, W, H + W))
    rho = (lap + ratio * lap.std()).astype(np.float32)
    img, st = _solve(rho, 0.0)
    f = rho.astype(np.float64)
    f -= f.mean()
    ref = O.poisson_neumann(f[None], [0.0])[0]
    assert st["status"] == 0 and 0.0 < st["rel_residual"] <= 1e-6, st
    assert np.abs(img - ref).max() <= TOL * (ref.max() - ref.min())
    left = np.linalg.norm(f - _laplacian(img)) / np.linalg.norm(f)
    ulp = 8.0 * np.abs(img).max() * 2.0 ** -24 * np.sqrt(f.size) / np.linalg.norm(f)
    assert left <= st["rel_residual"] + ulp
    np.testing.assert_allclose(st["rho_norm"], np.linalg.norm(f), rtol=1e-4)


@pytest.mark.parametrize("hw", [(97, 101), (128, 128), (757, 1355)])
@pytest.mark.parametrize("value", [0.1, 1.0 / 3.0, -1e5])
def test_constant_field_is_its_mean(hw, value):
    """Least squares: nothing is left of a constant field, whatever its FP32 sum rounds to."""
    rho = np.full(hw, value, np.float32)
    img, st = _solve(rho, 0.25)
    assert st["status"] == 0 and st["cycles"] == 0 and np.all(img == 0.25), st


@pytest.mark.parametrize("hw", [(128, 200), (757, 1355)])
def test_constant_field_with_one_pixel_off(hw):
    H, W = hw
    rho = np.full(hw, 1.0 / 3.0, np.float32)
    rho[5, 7] = 0.5
    img, st = _solve(rho, 0.0)
    f = rho.astype(np.float64)
    ref = O.poisson_neumann((f - f.mean())[None], [0.0])[0]
    assert st["status"] == 0 and st["rel_residual"] <= 1e-6, st
    assert np.abs(img - ref).max() <= TOL * (ref.max() - ref.min())
