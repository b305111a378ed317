"""The direct solve by cosine transforms (csrc/fct.cu) against the exact DCT solution of the
FP32 Laplacian field it is given (_field: the divergence as the library rounds it) and
against the multigrid cycles, at the sides where its transforms change: lengths of two,
three and four radices, the shortest ones, odd sides and primes (Bluestein), odd numbers
of rows (a row pair with one row), widths that are not a multiple of 4, one side past the
longest FFT (the multigrid takes those), thin images.

Tolerance: the image is stored in FP32 (half an ulp of its largest value) and the iterate
solves the system to a relative residual r <= 1e-6 whose remaining error is the rounding
of the transforms of the second cycle; its forward transform's white rounding noise,
2^-24 of the first cycle's residual, is amplified by at most the condition number 8 / lambda_min
of the grid, which for sides up to 4100 is 8 * (4100 / pi)^2 = 1.4e7, i.e. by less than one: the
second cycle's error is below the first residual's share of the image, 1e-5 of its range.
"""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2405_05446_gb300 as G

from gpu_util import ensure_lib, gpu_poisson

pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def _maps(C, H, W, seed):
    rng = np.random.default_rng(seed)
    y, x = np.mgrid[0:H, 0:W]
    img = np.stack([0.5 + 0.3 * np.sin(5.0 * x / W + c) * np.cos(4.0 * y / H) + 0.2 * (x > (0.3 + 0.1 * c) * W)
                    for c in range(C)]) + 0.02 * rng.standard_normal((C, H, W))
    return O.forward_gradients(img).astype(np.float32)


def _field(maps):
    """The divergence in FP32, its terms added in the library's order: the field the solve
    gets. Its rounding (1e-9 per pixel, white) is not the solver's: in the lowest mode of a
    64 x 4096 image it is worth 4e-5 of the image."""
    gx, gy = maps[:, 0], maps[:, 1]
    rho = np.zeros_like(gx)
    rho[:, :, :-1] += gx[:, :, :-1]
    rho[:, :, 1:] -= gx[:, :, :-1]
    rho[:, :-1, :] += gy[:, :-1, :]
    rho[:, 1:, :] -= gy[:, :-1, :]
    assert rho.dtype == np.float32
    return rho.astype(np.float64)


def _profiled(maps, mean, sopts=None):
    """The solve again under the profiler, which names the passes."""
    G.profile_begin()
    gpu_poisson(maps, mean, sopts)
    return G.profile_end()


@pytest.mark.parametrize("hw", [(32, 32), (33, 64), (97, 101), (64, 4096), (4096, 40), (48, 4095), (61, 2049),
                                (270, 480), (271, 482), (513, 257), (360, 1100), (12, 90)])
def test_direct_solve_matches_dct_oracle(hw):
    H, W = hw
    C = 3 if H * W < 100000 else 1
    mean = [0.5, 0.1, -0.2][:C]
    maps = _maps(C, H, W, H * 10007 + W)
    img, st = gpu_poisson(maps, mean)
    ref = O.poisson_neumann(_field(maps), mean)
    assert st["status"] == 0 and st["rel_residual"] <= 1e-6 and 1 <= st["cycles"] <= 3, st
    assert np.abs(img - ref).max() <= TOL * max(1.0, ref.max() - ref.min())
    np.testing.assert_allclose(img.mean(axis=(1, 2)), mean, atol=1e-6)
    assert "fct_columns" in _profiled(maps, mean)


@pytest.mark.parametrize("hw", [(40, 4097), (2, 2), (1, 130)])
def test_sides_outside_the_transforms_keep_the_multigrid(hw):
    H, W = hw
    maps = _maps(1, H, W, 3)
    assert "fct_columns" not in _profiled(maps, [0.5])


@pytest.mark.parametrize("hwc,direct", [((2061, 2176, 1), True), ((2061, 2176, 3), False), ((2061, 2175, 3), True),
                                        ((2153, 2560, 3), True), ((2153, 3840, 3), False), ((2160, 3840, 3), True)])
def test_large_sides_without_a_length_of_their_own(hwc, direct):
    """Even widths: both sides by Bluestein above 8M values, one of them above 22M, stay with
    the multigrid; either way the solve meets rtol."""
    H, W, C = hwc
    rho = torch.randn((C, H, W), device="cuda", generator=torch.Generator("cuda").manual_seed(H + W))
    rho -= rho.mean(dim=(1, 2), keepdim=True)
    img = torch.empty_like(rho)
    ws = torch.empty(G.workspace_size(0, C, W, H, None, None), dtype=torch.uint8, device="cuda")
    G.profile_begin()
    G.poisson_reconstruct_rho(rho, [0.5] * C, img, ws)
    names = G.profile_end()
    st = G.sync_status(ws)
    assert st["status"] == 0 and ("fct_columns" in names) == direct, (st, list(names))


@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("hw", [(150, 210), (101, 67)])
def test_direct_and_multigrid_agree_over_the_options(hw, storage):
    """Mask, threshold, storage format and a field whose sum is not zero: the default
    options take the direct solve, a caller's own coarsest grid the multigrid cycles."""
    H, W = hw
    rng = np.random.default_rng(H + storage)
    rho = rng.laplace(0, 0.05, (2, H, W)).astype(np.float32) + np.float32(0.01)
    mask = (rng.random(((H + 15) // 16, (W + 15) // 16)) < 0.7).astype(np.uint8)
    mean = [0.5, -0.25]
    out = []
    for coarse in (8, 9):
        so = G.solver_opts(storage=storage, coarse_max_dim=coarse, rho_threshold=0.03)
        ws = torch.empty(G.workspace_size(0, 2, W, H, None, so), dtype=torch.uint8, device="cuda")
        img = torch.empty((2, H, W), device="cuda")
        G.poisson_reconstruct_rho(torch.as_tensor(rho).cuda(), mean, img, ws, mask=torch.as_tensor(mask).cuda(), sopts=so)
        st = G.sync_status(ws)
        assert st["status"] == 0, st
        out.append((img.cpu().numpy().astype(np.float64), st))
    on = np.kron(mask, np.ones((16, 16)))[:H, :W] > 0
    field = np.where(on, rho, 0.0).astype(np.float64)
    ref = O.poisson_neumann(np.where(np.abs(field) >= np.float32(0.03), field, 0.0), mean)
    scale = ref.max() - ref.min()
    assert np.abs(out[0][0] - ref).max() <= TOL * scale
    assert np.abs(out[0][0] - out[1][0]).max() <= 1e-4 * scale  # the multigrid's rtol = 1e-6
    assert out[0][1]["rel_residual"] <= 1e-6 and out[0][1]["cycles"] < out[1][1]["cycles"]


def test_direct_solve_cycle_limits_and_status():
    """One cycle only: the residual is above a tight rtol and reported; a loose rtol is met.
    A zero field stops at once, a NaN is reported."""
    maps = _maps(1, 120, 200, 5)
    _, st = gpu_poisson(maps, [0.5], G.solver_opts(max_cycles=1, rtol=1e-9))
    assert st["status"] == G._abi.ERR_NO_CONVERGE and st["cycles"] == 1 and 1e-9 < st["rel_residual"] < 1e-4
    _, st = gpu_poisson(maps, [0.5], G.solver_opts(max_cycles=1, rtol=1e-4))
    assert st["status"] == 0 and st["cycles"] == 1
    img, st = gpu_poisson(np.zeros_like(maps), [0.25])
    assert st["status"] == 0 and st["cycles"] == 0 and np.all(img == 0.25)
    maps[0, 0, 3, 3] = np.nan
    _, st = gpu_poisson(maps, [0.5])
    assert st["status"] == G._abi.ERR_NONFINITE


@pytest.mark.parametrize("first", range(0, 4096, 512))
def test_every_side_runs_as_rows_and_as_columns(first):
    """Every side from 32 that the transforms take, as the width and as the height of a thin
    image: each pass is launched within its shared memory and the solve meets rtol."""
    rng = np.random.default_rng(first)
    img = torch.empty((1, 40 * 4096), device="cuda")
    for n in range(max(32, first + 1), first + 513):
        rho = torch.as_tensor(rng.standard_normal((1, 40 * n)).astype(np.float32)).cuda()
        rho -= rho.mean()
        for W, H in ((n, 40), (40, n)):
            ws = torch.empty(G.workspace_size(0, 1, W, H, None, None), dtype=torch.uint8, device="cuda")
            G.poisson_reconstruct_rho(rho.view(1, H, W), [0.5], img[:, :W * H].view(1, H, W), ws)
            st = G.sync_status(ws)
            assert st["status"] == 0 and st["rel_residual"] <= 1e-6, (W, H, st)
