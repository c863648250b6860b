"""The stored volume: field kernel, z-pair layout and free-corner mask.

Every grid below ends a pair of rows or slices, a warp of columns or a mask
word somewhere else. The exported volume has to equal, bit for bit, the same
single-rounded FP32 operations in numpy (and their halves on FP16 storage):
no tolerance. Marches through dense fields (the loop without the mask) and
half-empty ones (the loop with it) are held to the oracle, and a volume beyond
4 GiB to a closed form.
"""
import numpy as np
import pytest

import hh_inputs as hi
from parity_util import assert_parity_conditioned, export_volume, f32, gpu_trace

pytestmark = pytest.mark.gpu

DIMS = [(2, 2, 2), (3, 2, 5), (2, 3, 4), (5, 7, 9), (30, 6, 17), (31, 9, 16), (33, 32, 15),
        (62, 5, 34), (65, 4, 3), (14, 40, 33)]
K = np.float32(hi.K_GD)


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    from paper_2603_02048_gb300 import hh

    return hh, torch


def _density(dims, dense):
    nx, ny, nz = dims
    g = np.random.default_rng(nx * 10007 + ny * 101 + nz)
    rho = g.uniform(0.5, 2.5, size=(nz, ny, nx)).astype(np.float32)
    if not dense:  # a ball of matter, the rest exactly empty
        z, y, x = hi.voxel_centres(dims)
        r = ((x / nx - 0.3) ** 2 + (y / ny - 0.6) ** 2 + (z / nz - 0.4) ** 2) ** 0.5
        rho[np.broadcast_to(r > 0.3, rho.shape)] = 0.0
    return rho


def _field32(rho):
    """{dn, g} in FP32, one rounding per operation, as the kernel does them."""
    dn = (K * rho).astype(np.float32)
    out = np.empty(rho.shape + (4,), np.float32)
    out[..., 0] = dn
    for c, ax in ((1, 2), (2, 1), (3, 0)):
        n = rho.shape[ax]
        i = np.arange(n)
        lo, hi_ = np.take(dn, np.maximum(i - 1, 0), ax), np.take(dn, np.minimum(i + 1, n - 1), ax)
        f = np.where((i > 0) & (i < n - 1), np.float32(0.5), np.float32(1.0)).astype(np.float32)
        shape = [1, 1, 1]
        shape[ax] = n
        out[..., c] = (hi_ - lo) * f.reshape(shape)
    return out


@pytest.mark.parametrize("dense", [True, False])
@pytest.mark.parametrize("dims", DIMS)
def test_field_is_exact(gpu, dims, dense):
    hh, torch = gpu
    rho = _density(dims, dense)
    want = _field32(rho)
    rho_t = torch.from_numpy(rho.ravel()).cuda()
    for storage in ("fp32", "fp16"):
        vol = hh.hh_volume_from_density(rho_t, hh.make_grid(dims, 2.0, storage), float(K))
        got = export_volume(hh, torch, vol, dims).astype(np.float32)
        if storage == "fp32":
            assert np.array_equal(got, want)
        else:
            s = np.array(hh.hh_volume_scales(vol), np.float32)[[0, 1, 1, 1]]
            assert np.array_equal(got, (want / s).astype(np.float16).astype(np.float32) * s)
        vol.close()


@pytest.mark.parametrize("dims", DIMS)
def test_noalloc_field_is_exact(gpu, dims):
    """The same kernel on the caller's x-fastest buffer (an empty particle set
    plus one particle: the rest of the volume is exactly zero)."""
    hh, torch = gpu
    parts = torch.tensor([[d * 0.45 for d in dims] + [1.5]], device="cuda")
    grid = hh.make_grid(dims, 1.0)
    rho = torch.empty(dims[0] * dims[1] * dims[2], device="cuda")
    hh.hh_splat_density(parts, grid, rho)
    out = torch.full((4 * rho.numel(),), float("nan"), device="cuda")
    hh.hh_build_index_field_noalloc(parts, grid, float(K), out)
    want = _field32(rho.cpu().numpy().reshape(dims[::-1]))
    assert np.array_equal(out.cpu().numpy().reshape(want.shape), want)


@pytest.mark.parametrize("stepper", ["euler", "rk4"])
@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("dims,dense", [((31, 9, 16), True), ((14, 40, 33), True),
                                        ((33, 32, 15), False), ((30, 29, 31), False)])
def test_march_with_and_without_mask(gpu, oracle_lib, dims, dense, storage, stepper):
    hh, torch = gpu
    bg = hi.checker_background()
    bg_t = torch.from_numpy(bg).cuda()
    vol = hh.hh_volume_from_density(torch.from_numpy(_density(dims, dense).ravel()).cuda(),
                                    hh.make_grid(dims, 2.0, storage), float(K) * 0.1)
    vol4 = export_volume(hh, torch, vol, dims)
    cams = f32([hi.orbit_camera(dims, az, el, 37, 23, dist_factor=1.2)
                for az, el in ((0.0, 0.0), (110.0, 25.0), (200.0, -40.0))])
    params = f32(hi.params_rk4_fixed(dims, 0.5))
    params["stepper"] = stepper
    got = gpu_trace(hh, torch, vol, cams, params, bg_t)
    for cam, g in zip(cams, got):
        ref = oracle_lib.trace_grid(vol4, cam, params, bg)
        assert_parity_conditioned(g, ref, oracle_lib, {"kind": "grid", "vol4": vol4}, dims, cam,
                                  params)
    vol.close()


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("gap", [1, 2, 5, 9])
def test_march_in_and_out_of_free_cells(gpu, oracle_lib, storage, gap):
    """Shells of matter with gaps of `gap` voxels between them: rays change between
    samples that read zero, which go on asking the mask, and ones that do not."""
    hh, torch = gpu
    dims = (41, 36, 33)
    g = np.random.default_rng(gap)
    z, y, x = hi.voxel_centres(dims)
    r = np.sqrt((x - 20.0) ** 2 + (y - 18.0) ** 2 + (z - 16.0) ** 2)
    dn = np.where(r % (2 * gap + 2) < gap + 2, -3e-5 * (1 + 0.2 * g.random(r.shape)), 0.0)
    dn = dn.astype(np.float32)
    bg = hi.checker_background()
    bg_t = torch.from_numpy(bg).cuda()
    vol = hh.hh_volume_from_dn(torch.from_numpy(dn.ravel()).cuda(), hh.make_grid(dims, 1.0, storage))
    vol4 = export_volume(hh, torch, vol, dims)
    cams = f32([hi.orbit_camera(dims, 25.0, 15.0, 37, 23), hi.orbit_camera(dims, 160.0, -40.0, 21, 29)])
    adaptive = f32(hi.params_euler_adaptive(dims, theta_max=3e-3))
    fixed = f32(hi.params_rk4_fixed(dims, 0.5))
    fixed["stepper"] = "euler"
    for params in (adaptive, fixed):
        for cam, g in zip(cams, gpu_trace(hh, torch, vol, cams, params, bg_t)):
            ref = oracle_lib.trace_grid(vol4, cam, params, bg)
            assert_parity_conditioned(g, ref, oracle_lib, {"kind": "grid", "vol4": vol4}, dims, cam,
                                      params)
    vol.close()


def test_volume_beyond_4_gib(gpu):
    """dn = c x in the far half of a grid whose FP32 volume exceeds 4 GiB, rays
    along -z from the far corner, all their samples beyond the 4 GiB: the
    gradient is the same everywhere there, so Eq. 16 turns every ray by
    c ds (1 - w_x^2) / n a step. An offset that wrapped at 2^32 would read the
    empty half."""
    hh, torch = gpu
    dims, c, steps, h = (8, 4400, 4400), 1e-5, 60, 0.5
    dn = torch.zeros((dims[2], dims[1], dims[0]), device="cuda")
    dn[dims[2] // 2:, dims[1] // 2:] = (torch.arange(dims[0], device="cuda") + 0.5) * c
    vol = hh.hh_volume_from_dn(dn.view(-1), hh.make_grid(dims))
    del dn
    cam = f32({"eye": [4.0, 4390.0, 4390.0], "look_at": [4.0, 4390.0, 4300.0],
               "up": [0.0, 1.0, 0.0], "vfov_deg": 0.05, "width": 8, "height": 4})
    params = f32(hi.params_rk4_fixed(dims, h))
    params["stepper"] = "euler"
    bg_t = torch.from_numpy(hi.checker_background()).cuda()
    primary, got = (gpu_trace(hh, torch, vol, [cam], dict(params, max_steps=m), bg_t)[0]
                    for m in (0, steps))
    assert np.all(got["steps"] == steps)
    turn = got["exit_dir"][:, 0] - primary["exit_dir"][:, 0]
    # n - 1 is at most 8 c and w_x at most 9e-4 + 3e-4, so a step's turn is c h to
    # a relative 8 c + 2e-6 = 8.2e-5; FP32 adds 60 roundings of 3e-4
    want = steps * h * c
    assert np.abs(turn - want).max() <= want * (8.2e-5 + 60 * 2.0**-24)
    vol.close()


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("dims", [(70, 35, 50), (32, 46, 31), (33, 80, 47)])
def test_rebuild_leaves_nothing_behind(gpu, dims, storage):
    """Rebuilt from particles whose supports share no voxel (every density value
    is then one product, the same in every run), after a build that filled the
    whole volume and an empty one: bit for bit the volume and the rays of a
    fresh build."""
    hh, torch = gpu
    g = np.random.default_rng(sum(dims))
    h, kept = 1.0, []
    for _ in range(400):
        p = np.array([g.uniform(-2.0, n + 2.0) for n in dims])
        if all(np.abs(p - q).max() > 4 * h + 1 for q in kept):
            kept.append(p)
    parts = np.concatenate([kept, g.uniform(0.5, 2.0, (len(kept), 1))], 1).astype(np.float32)
    parts_t = torch.from_numpy(parts).cuda()
    grid = hh.make_grid(dims, h, storage)
    bg_t = torch.from_numpy(hi.checker_background()).cuda()
    cams = f32([hi.orbit_camera(dims, az, 20.0, 48, 40, dist_factor=0.9) for az in (0.0, 215.0)])
    params = f32(hi.params_rk4_fixed(dims, 0.5))
    params["stepper"] = "euler"
    fresh = hh.hh_build_index_field(parts_t, grid, 1e-4)
    want4 = export_volume(hh, torch, fresh, dims)
    want = gpu_trace(hh, torch, fresh, cams, params, bg_t)
    full = torch.full((dims[0] * dims[1] * dims[2],), 0.7, device="cuda")
    vol = hh.hh_volume_from_density(full, grid, 1.0)
    hh.hh_volume_rebuild(vol, parts_t[:0].contiguous(), 1e-4)
    assert not np.any(export_volume(hh, torch, vol, dims))
    hh.hh_volume_rebuild(vol, parts_t, 1e-4)
    assert np.array_equal(export_volume(hh, torch, vol, dims), want4)
    for a, b in zip(gpu_trace(hh, torch, vol, cams, params, bg_t), want):
        assert all(np.array_equal(a[n], b[n]) for n in a)
