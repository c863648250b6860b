"""The free-corner mask itself, and marches that use it.

A volume's mask has a bit per stored element, set when the cell that the
element is the first corner of reads eight zeros; a flag beside it says whether
marches ask it. Isolated strong voxels sit where the build's units end: columns
15/16 and 31 to 33 (a mask word's 16 columns, a word of nonzero bits), 63 to 65,
the first and last columns, rows and slices (copied into the halo), both rows
and slices of a pair. Every bit of a sampled cell is compared with numpy on the
exported volume, and rays through sparse volumes (the flag is set) are held to
the oracle.
"""
import ctypes
import itertools

import numpy as np
import pytest

import hh_inputs as hi
from parity_util import assert_parity_plain, export_volume, f32, gpu_trace

pytestmark = pytest.mark.gpu


class Record(ctypes.Structure):
    """The first members of a volume's host record (csrc/hh_internal.h)."""

    _fields_ = [("nx", ctypes.c_int), ("ny", ctypes.c_int), ("nz", ctypes.c_int),
                ("storage", ctypes.c_int), ("layout", ctypes.c_int), ("row", ctypes.c_uint),
                ("pair", ctypes.c_uint), ("h_kernel", ctypes.c_float), ("data", ctypes.c_void_p),
                ("bytes", ctypes.c_size_t), ("mask_off", ctypes.c_size_t),
                ("nz_words", ctypes.c_uint), ("free_dev", ctypes.c_void_p),
                ("nz_dev", ctypes.c_void_p), ("sparse_dev", ctypes.c_void_p)]


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    from paper_2603_02048_gb300 import hh

    return hh, torch


def _words(hh, torch, ptr, n):
    view = hh._DeviceArray(ptr, (n,), "<i4")
    return torch.as_tensor(view, device="cuda").cpu().numpy().view(np.uint32)


def _mask(hh, torch, vol, dims):
    """Bits of the sampled cells (nz + 1, ny + 1, nx + 1), and the flag."""
    nx, ny, nz = dims
    rec = ctypes.cast(vol.handle, ctypes.POINTER(Record)).contents
    assert (rec.nx, rec.ny, rec.nz, rec.nz_words) == (nx, ny, nz, (nx + 31) // 32)
    assert rec.data + rec.mask_off == rec.free_dev
    torch.cuda.synchronize()
    words = _words(hh, torch, rec.free_dev, (rec.pair * ((nz + 3) // 2) + 31) // 32)
    K, J, I = np.ogrid[:nz + 1, :ny + 1, :nx + 1]
    e = (K >> 1) * rec.pair + J * rec.row + 2 * I + (K & 1)
    return (words[e >> 5] >> (e & 31)) & 1, int(_words(hh, torch, rec.sparse_dev, 1)[0])


def _free(vol4):
    """The same from the exported volume."""
    p = np.pad(np.any(vol4 != 0.0, axis=-1), 1, mode="edge")
    busy = np.zeros(tuple(n - 1 for n in p.shape), bool)
    for k, j, i in itertools.product((0, 1), repeat=3):
        busy |= p[k:k + busy.shape[0], j:j + busy.shape[1], i:i + busy.shape[2]]
    return (~busy).astype(np.uint32)


def _spikes(dims, rate):
    picks = [sorted({g for g in (0, 1, 6, 14, 15, 16, 30, 31, 32, 33, 62, 63, 64, 65, n - 2, n - 1)
                     if 0 <= g < n}) for n in dims]
    rng = np.random.default_rng(sum(dims))
    dn = np.zeros(dims[::-1], np.float32)
    for x, y, z in itertools.product(*picks):
        if rng.random() < rate:
            dn[z, y, x] = rng.choice([-1.0, 1.0]) * rng.uniform(1e-3, 3e-3)
    return dn


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("dims", [(2, 2, 2), (6, 7, 33), (15, 34, 6), (16, 9, 17), (17, 33, 8),
                                  (31, 20, 9), (32, 5, 16), (33, 34, 20), (64, 3, 7), (65, 17, 18),
                                  (130, 6, 5)])
def test_mask_bits(gpu, dims, storage):
    hh, torch = gpu
    grid = hh.make_grid(dims, 2.0, storage)
    for rate in (0.02, 0.3):
        dn = _spikes(dims, rate)
        vol = hh.hh_volume_from_dn(torch.from_numpy(dn.ravel()).cuda(), grid)
        bits, _ = _mask(hh, torch, vol, dims)
        assert np.array_equal(bits, _free(export_volume(hh, torch, vol, dims)))
        vol.close()
    vol = hh.hh_volume_from_dn(torch.full((dn.size,), 1e-4, device="cuda"), grid)
    bits, sparse = _mask(hh, torch, vol, dims)
    assert not bits.any() and sparse == 0
    vol.close()


@pytest.mark.parametrize("stepper", ["euler", "rk4"])
@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("dims", [(33, 34, 20), (65, 17, 18)])
def test_marches_of_sparse_volumes(gpu, oracle_lib, dims, storage, stepper):
    hh, torch = gpu
    bg = hi.checker_background()
    bg_t = torch.from_numpy(bg).cuda()
    vol = hh.hh_volume_from_dn(torch.from_numpy(_spikes(dims, 0.05).ravel()).cuda(),
                               hh.make_grid(dims, 2.0, storage))
    _, sparse = _mask(hh, torch, vol, dims)
    assert sparse  # the march asks the mask
    vol4 = export_volume(hh, torch, vol, dims)
    assert np.count_nonzero(vol4[..., 0]) > 15
    cams = f32([hi.orbit_camera(dims, az, el, 64, 48, dist_factor=1.1)
                for az, el in ((0.0, 0.0), (90.0, 25.0), (200.0, -40.0), (315.0, 60.0))])
    params = f32(hi.params_rk4_fixed(dims, 0.5))
    params["stepper"] = stepper
    for cam, r in zip(cams, gpu_trace(hh, torch, vol, cams, params, bg_t)):
        ref = oracle_lib.trace_grid(vol4, cam, params, bg, nthreads=4)
        assert assert_parity_plain(r, ref, dims)["hits"] > 100
    vol.close()
