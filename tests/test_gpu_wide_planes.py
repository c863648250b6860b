"""Volumes whose planes are so wide that one pair of stored slices takes 4 GiB.

A cell whose first slice is the second of its pair then has its upper corners
beyond a 32-bit byte offset. Strong random values in a patch at the grid's
corner, rays through the patch across both grid slices (first slices of both
parities), single view, batch and server, each ray held to the oracle on the
patch.
"""
import numpy as np
import pytest

import hh_inputs as hi
from parity_util import assert_parity_plain, f32, gpu_trace

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stepper", ["euler", "rk4"])
@pytest.mark.parametrize("storage,dims", [("fp32", (16384, 8192, 2)), ("fp16", (16384, 16384, 2))])
def test_slice_pair_beyond_4_gib(oracle_lib, storage, dims, stepper):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    from paper_2603_02048_gb300 import hh

    nx, ny, nz = dims
    px, py = 48, 40  # the patch the rays see; zero in its outer 4 voxels
    g = np.random.default_rng(5)
    patch = np.zeros((nz, py, px), np.float32)
    patch[:, 4:-4, 4:-4] = g.uniform(-3e-3, 3e-3, (nz, py - 8, px - 8))
    dn = torch.zeros((nz, ny, nx), device="cuda")
    dn[:, :py, :px] = torch.from_numpy(patch).cuda()
    vol = hh.hh_volume_from_dn(dn.view(-1), hh.make_grid(dims, 2.0, storage))
    del dn
    out = torch.empty(nx * ny * nz * 4, device="cuda")
    hh.hh_volume_export(vol, out)
    torch.cuda.synchronize()
    vol4 = out.view(nz, ny, nx, 4)[:, :py, :px].cpu().numpy().astype(np.float64)
    del out
    assert np.count_nonzero(vol4[..., 0]) > 2000
    # 24 x 20 rays over 20 x 16 voxels of the patch's middle
    cams = f32([{"eye": [px / 2, py / 2, z], "look_at": [px / 2, py / 2, 1.0],
                 "up": [0.0, 1.0, 0.0], "vfov_deg": 30.0, "width": 24, "height": 20}
                for z in (-30.0, 32.0)])
    params = f32(hi.params_rk4_fixed((px, py, nz), 0.25))
    params["stepper"] = stepper
    bg = hi.checker_background()
    bg_t = torch.from_numpy(bg).cuda()
    got = gpu_trace(hh, torch, vol, cams, params, bg_t)
    outs = [{"rgb": torch.empty(24 * 20 * 3, device="cuda"),
             "exit_dir": torch.empty(24 * 20 * 3, device="cuda")} for _ in cams]
    b = hh.hh_batch_create(vol, cams, params, bg_t, outs)
    hh.hh_batch_launch(b)
    torch.cuda.synchronize()
    b.close()
    srv = hh.hh_serve_create(64 << 20, 2)
    hh.hh_serve_put_volume(srv, 0, vol)
    ticket = hh.hh_serve_submit(srv, 0, cams, params, bg_t, 1 | 2 | 4)
    hh.hh_serve_wait(srv, ticket, 20000)
    served = [hh.hh_serve_view(srv, ticket, i, 24, 20) for i in range(len(cams))]
    hh.hh_serve_release(srv, ticket)
    srv.close()
    for cam, r, o, v in zip(cams, got, outs, served):
        ref = oracle_lib.trace_grid(vol4, cam, params, bg, nthreads=4)
        assert np.all(ref["flags"] == 3)  # every ray enters the patch and leaves it
        assert_parity_plain(r, ref, (px, py, nz))
        want = r["exit_dir"].astype(np.float32)
        assert np.array_equal(o["exit_dir"].cpu().numpy().reshape(-1, 3), want)
        assert np.array_equal(v["exit_dir"].cpu().numpy().reshape(-1, 3), want)
    vol.close()
