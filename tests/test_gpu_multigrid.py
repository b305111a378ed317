"""The multigrid cycles at full size. They serve sides above 4096, large even widths whose
sides have no transform of their own, and a caller's own omega or coarsest grid; with the
default options most sizes are solved directly (fct.cu). Here the tests of the parity file that
are about the cycles (16-bit storage, in-place levels, per-channel loops and their graphs,
the cached coarse factor) run once more with coarse_max_dim = 9, which builds the same levels
at these sizes and takes the cycles; the last ones compare the default routes that take them
with the oracle. Tolerances are those of the parity file."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2405_05446_gb300 as G

import test_gpu_parity as P
from gpu_util import IMG_TOL, ensure_lib, gpu_poisson, img_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


@pytest.fixture
def cycles(monkeypatch):
    """Every default option structure asks for a coarsest grid of 9."""
    make = G.solver_opts
    opts = lambda **kw: make(**{"coarse_max_dim": 9, **kw})  # noqa: E731
    monkeypatch.setattr(G, "solver_opts", opts)
    for name in ("poisson_reconstruct", "poisson_reconstruct_rho", "render_view"):
        def call(*a, _f=getattr(G, name), _at={"render_view": 6}.get(name, 5), **kw):
            a = list(a)
            if len(a) > _at:
                a[_at] = a[_at] or opts()
            else:
                kw["sopts"] = kw.get("sopts") or opts()
            return _f(*a, **kw)
        monkeypatch.setattr(G, name, call)
    G.profile_begin()
    gpu_poisson(np.zeros((1, 2, 64, 96), np.float32) + np.float32(0.1), [0.5])
    names = G.profile_end()
    assert "mg0_up" in names and "fct_columns" not in names  # the cycles it is


@pytest.mark.parametrize("max_cycles", [1, 30])
def test_identical_channels(cycles, max_cycles):
    P.test_identical_channels_give_identical_images_1080p(max_cycles)


def test_channel_split(cycles):
    P.test_channel_split_equals_one_channel_solves()


@pytest.mark.parametrize("storage", ["bf16", "f16"])
def test_16bit_storage(cycles, storage):
    P.test_poisson_16bit_storage_reaches_tolerance_1080p(storage)
    P.test_render_view_16bit_storage(storage)


@pytest.mark.parametrize("storage", ["f32", "bf16", "f16"])
def test_storage_4k(cycles, storage):
    P.test_poisson_storage_4k_against_oracle(storage)


def test_storage_scaling(cycles):
    P.test_storage_scaling_keeps_fp32_bitwise()


def test_coarse_cache_across_sizes(cycles):
    P.test_poisson_coarse_cache_reused_across_sizes()


def test_graph_and_direct_loops(cycles):
    P.test_graph_and_direct_cycle_loops_agree()


def test_launch_count(cycles):
    P.test_kernel_launch_count_covers_graph_kernels()


def test_graph_cache_layouts(cycles):
    P.test_graph_cache_distinguishes_workspace_layouts()


def test_two_relaxations_share_a_workspace():
    """omega = 1 and 1.1, neither of them the direct solve's: a stale graph would repeat one."""
    rng = np.random.default_rng(21)
    C, H, W = 3, 270, 480
    maps = torch.as_tensor(rng.laplace(0, 0.1, (C, 2, H, W)).astype(np.float32)).cuda()
    ws = torch.empty(G.workspace_size(0, C, W, H, None, None), dtype=torch.uint8, device="cuda")
    img = []
    for omega in (1.0, 1.1, 1.0):
        out = torch.empty((C, H, W), device="cuda")
        G.poisson_reconstruct(maps, [0.5] * C, out, ws, sopts=G.solver_opts(omega=omega))
        assert G.sync_status(ws)["status"] == 0
        img.append(out.cpu().numpy().astype(np.float64))
    assert np.array_equal(img[0], img[2]) and not np.array_equal(img[0], img[1])
    ref = O.poisson_neumann(O.divergence(maps.cpu().numpy().astype(np.float64)), [0.5] * C)
    assert img_err(img[1], ref)[0] <= IMG_TOL


@pytest.mark.parametrize("hwc", [(1200, 4100, 1), (2061, 2176, 3)])
def test_default_routes_that_take_the_cycles(hwc):
    H, W, C = hwc
    rng = np.random.default_rng(H + W)
    maps = rng.laplace(0, 0.1, (C, 2, H, W)).astype(np.float32)
    mean = [0.5, 0.4, 0.6][:C]
    img, st = gpu_poisson(maps, mean)
    assert st["status"] == 0 and st["cycles"] > 3, st  # more than the direct solve has
    ref = O.poisson_neumann(O.divergence(maps.astype(np.float64)), mean)
    assert img_err(img, ref)[0] <= IMG_TOL


@pytest.mark.parametrize("hw", [(40, 4097), (4098, 60)])
def test_thin_default_routes_that_take_the_cycles(hw):
    """Thin images, where a relative residual of 1e-6 bounds no error (the condition number is
    1e7): the FP64 residual of the image itself, as for the parity file's strips."""
    H, W = hw
    img0 = np.random.default_rng(H).random((1, H, W))
    maps = O.forward_gradients(img0)
    rho = O.divergence(maps)
    img, st = gpu_poisson(maps.astype(np.float32), [0.5])
    assert st["status"] == 0 and st["rel_residual"] <= 1e-6 and st["cycles"] > 3, st
    assert np.linalg.norm(rho - O.laplacian_neumann(img)) <= 2e-6 * np.linalg.norm(rho)
    assert abs(img.mean() - 0.5) <= 1e-6
