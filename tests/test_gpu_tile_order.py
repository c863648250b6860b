"""Every tile of a view is marched exactly once, whatever row the launch starts
with: views whose volume centre projects above, below, inside and far outside
the image or lies behind the camera, with one to many rows of tiles, through the
single-view launch, both tile orders of the batch and both of its schedulings.
"""
import pytest

import hh_inputs as hi
from parity_util import f32


def test_row_orders_are_permutations():
    """The row that the single-view kernel takes i-th of n from row mid outwards
    (the rule restated: it covers every row once for every n and mid)."""
    def row_from(i, n, mid):
        if i <= 2 * min(mid, n - 1 - mid):
            return mid + ((i + 1) // 2 if i % 2 else -(i // 2))
        return i if mid < n - 1 - mid else n - 1 - i

    for n in range(1, 40):
        for mid in range(n):
            assert sorted(row_from(i, n, mid) for i in range(n)) == list(range(n))


@pytest.mark.gpu
@pytest.mark.parametrize("w,h", [(17, 1), (9, 8), (40, 9), (33, 24), (16, 61), (130, 100)])
def test_every_pixel_once(w, h):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    from paper_2603_02048_gb300 import hh

    dims = (24, 20, 28)
    vol = hh.hh_volume_from_dn(torch.from_numpy(hi.plume_dn_grid(dims=dims).ravel()).cuda(),
                               hh.make_grid(dims))
    bg_t = torch.from_numpy(hi.checker_background()).cuda()
    eye = [-30.0, 8.0, 12.0]
    cams = f32([{"eye": eye, "look_at": at, "up": [0.0, 0.0, 1.0], "vfov_deg": 50.0, "width": w,
                 "height": h} for at in ([12.0, 10.0, 14.0], [12.0, 10.0, 30.0], [12.0, 10.0, -15.0],
                                         [12.0, 10.0, 400.0], [-80.0, 8.0, 11.0])])
    params = f32(hi.params_rk4_fixed(dims, 0.5))
    params["stepper"] = "euler"
    # one view at a time: a pixel that no tile covers keeps its NaN
    single = []
    for cam in cams:
        out = [{"rgb": torch.full((3 * w * h,), float("nan"), device="cuda"),
                "steps": torch.full((w * h,), -1, dtype=torch.int32, device="cuda")}]
        hh.hh_trace(vol, [cam], params, bg_t, out)
        single.append(out[0])
        assert not torch.isnan(out[0]["rgb"]).any() and (out[0]["steps"] >= 0).all()
    for order, group, tile_w in ((0, 0, 8), (1, 0, 8), (1, 1, 4), (1, 0, 16)):
        outs = [{"rgb": torch.full((3 * w * h,), float("nan"), device="cuda")} for _ in cams]
        b = hh.hh_batch_create(vol, cams, params, bg_t, outs)
        hh.hh_batch_set_config(b, 64, 0, 32, tile_w, order, group)
        hh.hh_batch_launch(b)
        torch.cuda.synchronize()
        assert all(torch.equal(o["rgb"], s["rgb"]) for o, s in zip(outs, single))
        b.close()
    vol.close()
