"""Eq. 18 with a regulariser, a tolerance or steps so small that |g_perp|^2 or a
quotient's operands are FP32 subnormals: still the step Eq. 18 gives, counted
against the oracle. (A march that drops subnormals takes |g_perp| = 5e-20 for
zero and steps by h_max, and a subnormal tolerance for zero and steps by h_min.)
"""
import numpy as np
import pytest

import hh_inputs as hi
from parity_util import f32, gpu_trace

pytestmark = pytest.mark.gpu

# c: dn = c x; steps n theta / (c + eps) of 0.1961, 0.1953 and 0.2101 over 24
# voxels: 122.4, 122.9 and 114.2 of them, at least 0.15 from a whole number,
# where |g_perp|^2 = c^2 and theta are held to 6e-7 and the rest to 1e-6
CASES = [(5e-20, 1e-20, 1e-21), (0.0, 2.93e-39, 1.5e-38), (1.0e-19, 2.5e-20, 1.9e-20)]


@pytest.mark.parametrize("stepper", ["euler", "rk4"])
@pytest.mark.parametrize("c,theta,eps", CASES)
def test_step_count(oracle_lib, c, theta, eps, stepper):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    from paper_2603_02048_gb300 import hh

    dims = (12, 10, 24)
    x = hi.voxel_centres(dims)[2]
    dn = np.broadcast_to(c * x, dims[::-1]).astype(np.float32)
    vol4 = np.zeros(dims[::-1] + (4,))
    vol4[..., 0] = dn
    vol4[..., 1] = c
    bg = hi.checker_background()
    bg_t = torch.from_numpy(bg).cuda()
    cam = f32({"eye": [6.0, 5.0, -20.0], "look_at": [6.0, 5.0, 0.0], "up": [0.0, 1.0, 0.0],
               "vfov_deg": 0.05, "width": 8, "height": 4})
    params = f32({"stepper": stepper, "adaptive": True, "h_fixed": 1.0, "h_min": 0.01,
                  "h_max": 4.0, "theta_max": theta, "eps": eps, "max_steps": 4000})
    want = oracle_lib.trace_grid(vol4, cam, params, bg)
    assert np.all(want["flags"] == 3) and 100 < want["steps"].min() <= want["steps"].max() < 130
    vol = hh.hh_volume_from_dn(torch.from_numpy(dn.ravel().copy()).cuda(), hh.make_grid(dims))
    got = gpu_trace(hh, torch, vol, [cam], params, bg_t)[0]
    outs = [{"rgb": torch.empty(32 * 3, device="cuda"),
             "steps": torch.empty(32, dtype=torch.int32, device="cuda")}]
    b = hh.hh_batch_create(vol, [cam], params, bg_t, outs)
    for refill in (32, 8):
        hh.hh_batch_set_config(b, refill_min=refill)
        hh.hh_batch_launch(b)
        torch.cuda.synchronize()
        assert np.array_equal(outs[0]["steps"].cpu().numpy(), want["steps"])
    b.close()
    assert np.array_equal(got["steps"], want["steps"])
    assert np.array_equal(got["flags"], want["flags"])
    vol.close()
