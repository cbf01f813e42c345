"""Parity of the phantom generator, FDK and the gradient initialiser with the CPU oracle."""
import ctypes

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gsct():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2604_01844_gb300 as g
    from paper_2604_01844_gb300 import build

    build.build()
    return g


def _s():
    return torch.cuda.current_stream().cuda_stream


def test_phantom_project_and_voxelize(orc, gsct):
    B = gsct.binding
    ell = synth.ellipsoid_phantom(1, 40)
    W = H = 64
    views = synth.cone_views(6, W, H)
    d_ell = torch.from_numpy(ell.astype(np.float32)).cuda()
    d_views = gsct.views_to_device(views, "cuda")
    img = torch.empty((6, H, W), device="cuda")
    B.check(B.lib().gs_phantom_project(B.ptr(d_ell), 40, B.ptr(d_views), 6, W, H, B.ptr(img),
                                       _s()), "phantom_project")
    want = orc.phantom_project(ell.astype(np.float32).astype(np.float64), orc.views64(views), W, H)
    got = img.cpu().numpy()
    assert np.abs(got - want).max() <= 1e-4 * np.abs(want).max()
    grid = synth.cube_grid(48)
    vol = torch.empty((48, 48, 48), device="cuda")
    B.check(B.lib().gs_phantom_voxelize(B.ptr(d_ell), 40, ctypes.byref(B.grid_struct(grid)),
                                        B.ptr(vol), _s()), "phantom_voxelize")
    want_v = orc.phantom_voxelize(ell.astype(np.float32).astype(np.float64), grid)
    diff = np.abs(vol.cpu().numpy() - want_v) > 1e-5
    # only voxel centres on an ellipsoid surface (FP32 vs FP64 inside test) may differ
    assert diff.mean() < 1e-3


def test_fdk_matches_oracle(orc, gsct):
    from oracle.init import fdk
    B = gsct.binding
    ell = synth.ellipsoid_phantom(2, 10)
    W, H, nv = 64, 48, 24
    views = synth.cone_views(nv, W, H)
    V = orc.views64(views)
    proj = orc.phantom_project(ell, V, W, H).astype(np.float32)
    grid = synth.cube_grid(40)
    want = fdk(proj.astype(np.float64), V, grid)
    d_proj = torch.from_numpy(proj).cuda()
    d_views = gsct.views_to_device(views, "cuda")
    ws = torch.empty(B.lib().gs_fdk_workspace_size(nv, W, H), dtype=torch.uint8, device="cuda")
    vol = torch.empty((40, 40, 40), device="cuda")
    B.check(B.lib().gs_fdk(B.ptr(d_proj), B.ptr(d_views), nv, W, H,
                           ctypes.byref(B.grid_struct(grid)), B.ptr(vol), B.ptr(ws), ws.numel(),
                           _s()), "gs_fdk")
    got = vol.cpu().numpy()
    assert np.abs(got - want).max() <= 1e-4 * np.abs(want).max(), \
        float(np.abs(got - want).max() / np.abs(want).max())


@pytest.mark.parametrize("n", [1, 500, 4000])
def test_grad_init_matches_oracle(orc, gsct, n):
    from oracle.init import grad_init
    B = gsct.binding
    rng = np.random.default_rng(n)
    grid = synth.cube_grid(32)
    ell = synth.ellipsoid_phantom(3, 12)
    V = orc.phantom_voxelize(ell, grid).astype(np.float32)
    V += (0.01 * rng.standard_normal(V.shape)).astype(np.float32)
    u = rng.random((n, 4)).astype(np.float32)
    mr, sc, q, idx, margin = grad_init(V, grid, n, 0.05, 0.15, 1e-4, u)
    d_V = torch.from_numpy(V).cuda()
    d_u = torch.from_numpy(u).cuda()
    out = [torch.empty((n, 4), device="cuda") for _ in range(3)]
    vox = torch.empty(n, dtype=torch.int32, device="cuda")
    ws = torch.empty(B.lib().gs_grad_init_workspace_size(ctypes.byref(B.grid_struct(grid)), n),
                     dtype=torch.uint8, device="cuda")
    B.check(B.lib().gs_grad_init(B.ptr(d_V), ctypes.byref(B.grid_struct(grid)), n, 0.05, 0.15,
                                 1e-4, B.ptr(d_u), *[B.ptr(t) for t in out], B.ptr(vox),
                                 B.ptr(ws), ws.numel(), _s()), "gs_grad_init")
    got_idx = vox.cpu().numpy()
    safe = margin > 1e-12
    assert safe.mean() > 0.99
    assert np.array_equal(got_idx[safe], idx[safe])  # integer decision: bit-exact
    g_mr, g_sc, g_q = (t.cpu().numpy().astype(np.float64) for t in out)
    np.testing.assert_allclose(g_mr[safe, :3], mr[safe, :3], rtol=0, atol=1e-6)
    np.testing.assert_allclose(g_mr[safe, 3], mr[safe, 3], rtol=1e-5, atol=1e-6)
    if n > 1:
        np.testing.assert_allclose(g_sc[safe, 0], sc[safe, 0], rtol=1e-4, atol=1e-6)
    assert np.all(g_q[:, 0] == 1) and np.all(g_q[:, 1:] == 0)


# detectors that no filter tile divides (16 outputs, 8 rows; the wide form above 2,700 columns),
# volumes at the edges of the 16 x 16 blocks and of each voxels-per-thread choice, frames with a
# component along z (the general back-projection)
@pytest.mark.parametrize("nv,W,H,dims,tilt", [(1, 1, 1, (5, 4, 3), 0.0), (5, 17, 9, (17, 15, 23), 0.0),
                                              (6, 97, 41, (33, 16, 47), 0.2),
                                              (2, 2801, 6, (24, 20, 18), 0.1),
                                              (70, 64, 48, (96, 80, 64), 0.0)])
def test_fdk_ragged_and_tilted(orc, gsct, nv, W, H, dims, tilt):
    """1e-4 of the peak as for images and volumes, plus the rounding of a detector position (about
    2.5 x 2^-24 of the side) times the steepest slope, twice the peak per pixel."""
    from oracle.init import fdk
    B = gsct.binding
    views = synth.cone_views(nv, W, H)
    if tilt:
        for v in views:
            n = v["det_center"] - v["src"]
            n = n / np.linalg.norm(n) + np.array([0, 0, tilt])
            n /= np.linalg.norm(n)
            pitch = np.linalg.norm(v["v"])
            u = np.cross([0, 0, 1], n)
            u /= np.linalg.norm(u)
            w = np.cross(n, u)
            v["src"], v["det_center"] = -4 * n, 2 * n
            v["u"] = pitch * (np.cos(0.3) * u + np.sin(0.3) * w)
            v["v"] = pitch * (np.cos(0.3) * w - np.sin(0.3) * u)
    rng = np.random.default_rng(W)
    proj = (1 + rng.random((nv, H, W))).astype(np.float32)
    grid = synth.cube_grid(8)
    grid["dims"] = dims
    # the whole detector and some voxels outside it
    half = 2.2 * min(W, H) / max(W, H)
    grid["voxel"] = [half / d for d in dims]
    grid["origin"] = [-half / 2] * 3
    want = fdk(proj.astype(np.float64), orc.views64(views), grid)
    d_proj, d_views = torch.from_numpy(proj).cuda(), gsct.views_to_device(views, "cuda")
    ws = torch.full((B.lib().gs_fdk_workspace_size(nv, W, H),), 255, dtype=torch.uint8, device="cuda")
    vol = torch.full(dims[::-1], float("nan"), device="cuda")
    B.check(B.lib().gs_fdk(B.ptr(d_proj), B.ptr(d_views), nv, W, H,
                           ctypes.byref(B.grid_struct(grid)), B.ptr(vol), B.ptr(ws), ws.numel(),
                           _s()), "gs_fdk")
    assert np.abs(want).max() > 0
    tol = 1e-4 + 2.0 ** -21 * max(W, H)
    assert np.abs(vol.cpu().numpy() - want).max() <= tol * np.abs(want).max()


@pytest.mark.parametrize("offset", [4, 8, 12])
def test_fdk_workspace_at_any_address(orc, gsct, offset):
    """A workspace that starts between 16-byte boundaries: the same volume, and not a byte written
    outside the size asked for."""
    B = gsct.binding
    nv, W, H, dims = 3, 37, 21, (9, 10, 11)
    grid = synth.cube_grid(16)
    grid["dims"] = dims
    d_views = gsct.views_to_device(synth.cone_views(nv, W, H), "cuda")
    proj = torch.rand((nv, H, W), device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    size = B.lib().gs_fdk_workspace_size(nv, W, H)
    vols = []
    for off in (0, offset):
        room = torch.full((size + 64,), 171, dtype=torch.uint8, device="cuda")
        vol = torch.empty(tuple(reversed(dims)), device="cuda")
        B.check(B.lib().gs_fdk(B.ptr(proj), B.ptr(d_views), nv, W, H,
                               ctypes.byref(B.grid_struct(grid)), B.ptr(vol), B.ptr(room) + off, size,
                               _s()), "gs_fdk")
        assert bool((room[:off] == 171).all()) and bool((room[off + size:] == 171).all())
        vols.append(vol)
    assert torch.equal(vols[0], vols[1])


@pytest.mark.parametrize("axis", [0, 2])
def test_fdk_of_the_longest_line(orc, gsct, axis):
    """2^31 - 1 voxels in one line, the most an int holds: every voxel is written, and the last one
    holds what a single voxel there holds (1e-4 of it, as for volumes)."""
    B = gsct.binding
    nv, W, H = 2, 16, 16
    d_views = gsct.views_to_device(synth.cone_views(nv, W, H), "cuda")
    proj = torch.ones((nv, H, W), device="cuda")
    ws = torch.empty(B.lib().gs_fdk_workspace_size(nv, W, H), dtype=torch.uint8, device="cuda")

    def run(dims, origin, voxel):
        grid = synth.cube_grid(8)
        grid["dims"], grid["origin"], grid["voxel"] = dims, origin, voxel
        vol = torch.full((int(np.prod(dims, dtype=np.int64)),), float("nan"), device="cuda")
        B.check(B.lib().gs_fdk(B.ptr(proj), B.ptr(d_views), nv, W, H,
                               ctypes.byref(B.grid_struct(grid)), B.ptr(vol), B.ptr(ws), ws.numel(),
                               _s()), "gs_fdk")
        return vol

    n, origin, voxel = 2 ** 31 - 1, [0.0, 0.0, 0.0], [1e-3] * 3
    dims = [1, 1, 1]
    dims[axis], voxel[axis] = n, 0.5 / n
    line = run(dims, origin, voxel)
    origin[axis], voxel[axis] = 0.5 - 1e-6, 2e-6
    one = run([1, 1, 1], origin, voxel)
    assert not bool(torch.isnan(line).any())
    assert float(one) != 0 and abs(float(line[-1]) - float(one)) <= 1e-4 * abs(float(one))
