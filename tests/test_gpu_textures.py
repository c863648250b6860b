"""Textures of odd sizes at every byte offset: the same image as from an aligned
copy, bit for bit, and the oracle's, with rays on the first and the last texel
(the map's poles, a plane's corners)."""
import numpy as np
import pytest

import hh_inputs as hi
from parity_util import assert_parity_plain, f32, gpu_trace

pytestmark = pytest.mark.gpu


def _defined(ref):
    """Rays that see something definite: not the board's very edge (where the last
    bit decides between it and the map), not the map's very pole (any azimuth)."""
    p, d = ref["exit_pos"], ref["exit_dir"]
    with np.errstate(all="ignore"):
        t = (20.0 - p[:, 0]) / d[:, 0]
        at = p[:, 1:] + t[:, None] * d[:, 1:]
        out = np.max(np.abs(at - 4.0), axis=1) - 4.0  # beyond the board's outline
        edge = (np.abs(out) < 1e-9) & (t > 0)
    return ~edge & (np.hypot(d[:, 0], d[:, 1]) > 1e-9)


@pytest.mark.parametrize("size", [(1, 2), (2, 2), (5, 3), (7, 5)])
def test_unaligned_textures(oracle_lib, size):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    from paper_2603_02048_gb300 import hh

    W, H = size
    g = np.random.default_rng(10 * W + H)
    env = g.integers(0, 256, (H, W, 3), dtype=np.uint8)
    tex = g.integers(0, 256, (max(H, 3), max(W, 3), 3), dtype=np.uint8)
    dims = (8, 8, 8)
    plane = {"origin": [20.0, 0.0, 0.0], "u": [0.0, 8.0, 0.0], "v": [0.0, 0.0, 8.0], "tex": tex}
    vol = hh.hh_volume_from_dn(torch.zeros(512, device="cuda"), hh.make_grid(dims))
    # at the board, and at both poles of the map
    cams = f32([{"eye": [-9.0, 4.0, 4.0], "look_at": [20.0, 4.0, 4.0], "up": [0.0, 0.0, 1.0],
                 "vfov_deg": 20.0, "width": 41, "height": 33}] +
               [{"eye": [4.0, 4.0, 4.0 - 20 * s], "look_at": [4.0, 4.0, 4.0], "up": [1.0, 0.0, 0.0],
                 "vfov_deg": 150.0, "width": 41, "height": 33} for s in (1, -1)])
    params = f32(hi.params_rk4_fixed(dims, 0.5))

    def at_offset(a, off):
        buf = torch.zeros(a.size + 16, dtype=torch.uint8, device="cuda")
        view = buf[off:off + a.size].view(a.shape)
        view.copy_(torch.from_numpy(a))
        return view

    images = []
    for off in range(4):
        scene = (at_offset(env, off), [dict(plane, tex=at_offset(tex, 3 - off))])
        images.append(gpu_trace(hh, torch, vol, cams, params, scene))
        for cam, r in zip(cams, images[-1]):
            ref = oracle_lib.trace_grid(np.zeros(dims + (4,)), cam, params, env, planes=[plane])
            sel = np.flatnonzero(_defined(ref))
            assert len(sel) >= 41 * 33 - 3  # both sides of the board, and the pole
            assert_parity_plain(r, {k: v[sel] for k, v in ref.items()}, dims, sel)
    for other in images[1:]:
        for a, b in zip(images[0], other):
            assert np.array_equal(a["rgb"], b["rgb"])
    vol.close()
