"""Chains of dependent launches (clear, splat, field, mask, march) on one stream.

Each kernel's blocks may start before the kernel ahead of it ends. Frames
enqueued back to back have to give, bit for bit, what the same calls give with
a synchronisation after each, on a stream and replayed from a captured graph.
The particles' supports do not overlap, so no sum depends on an order.
"""
import numpy as np
import pytest

import hh_inputs as hi

pytestmark = pytest.mark.gpu

DIMS = (83, 61, 47)


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    from paper_2603_02048_gb300 import hh

    return hh, torch


def _particles(torch, h, seed):
    """A lattice wider than the support, some of its places taken."""
    g = np.random.default_rng(seed)
    axes = [np.arange(2 * h + 1, n - 2 * h - 1, 4 * h + 1) for n in DIMS]
    at = np.stack(np.meshgrid(*axes, indexing="ij"), axis=-1).reshape(-1, 3)
    at = at[g.random(len(at)) < 0.6] + g.uniform(-0.4, 0.4, 3)
    m = g.uniform(0.5, 2.0, (len(at), 1))
    return torch.from_numpy(np.concatenate([at, m], axis=1).astype(np.float32)).cuda()


def _setup(hh, torch, storage, h):
    parts = [_particles(torch, h, s) for s in range(3)]
    parts.append(parts[0][:0])  # an empty frame
    vol = hh.hh_build_index_field(parts[0], hh.make_grid(DIMS, h, storage), 2.26e-4)
    cams = [hi.orbit_camera(DIMS, a, 15.0, 97, 61) for a in (20.0, 200.0)]
    params = hi.params_euler_adaptive(DIMS, theta_max=3e-5)
    bg = torch.from_numpy(hi.checker_background()).cuda()

    def frame(p, outs):
        hh.hh_volume_rebuild(vol, p, 2.26e-4)
        hh.hh_trace(vol, cams, params, bg, outs)

    def buffers():
        return [{"rgb": torch.zeros(97 * 61 * 3, device="cuda"),
                 "exit_dir": torch.zeros(97 * 61 * 3, device="cuda")} for _ in cams]

    return parts, frame, buffers


def _wanted(torch, parts, frame, buffers):
    want = []
    for p in parts:
        outs = buffers()
        frame(p, outs)
        torch.cuda.synchronize()
        want.append(outs)
    assert not torch.equal(want[0][0]["exit_dir"], want[1][0]["exit_dir"])
    return want


def _equal(torch, got, want):
    for g, w in zip(got, want):
        for k in w:
            assert torch.equal(g[k], w[k])


@pytest.mark.parametrize("h", [1.0, 2.0, 5.0])  # 5: the wide splat kernel
@pytest.mark.parametrize("storage", ["fp32", "fp16"])
def test_frames_back_to_back(gpu, storage, h):
    hh, torch = gpu
    parts, frame, buffers = _setup(hh, torch, storage, h)
    want = _wanted(torch, parts, frame, buffers)
    got = [buffers() for _ in range(24)]
    torch.cuda.synchronize()
    for i, outs in enumerate(got):
        frame(parts[i % 4], outs)
    torch.cuda.synchronize()
    for i, outs in enumerate(got):
        _equal(torch, outs, want[i % 4])


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("fork", [False, True])
def test_captured_frames(gpu, storage, fork):
    """Frames captured into one graph (the odd ones on a second stream, joined by
    events), replayed with other particles in the same buffers."""
    hh, torch = gpu
    parts, frame, buffers = _setup(hh, torch, storage, 2.0)
    n = min(len(p) for p in parts[:3])
    sets = [p[:n].clone() for p in parts[:3]]
    want = _wanted(torch, sets, frame, buffers)
    empty = buffers()
    frame(parts[3], empty)
    held, outs, side = sets[0].clone(), [buffers() for _ in range(4)], torch.cuda.Stream()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        main = torch.cuda.current_stream()
        for i, o in enumerate(outs):
            p = parts[3] if i == 2 else held
            if fork and i % 2:
                side.wait_stream(main)
                with torch.cuda.stream(side):
                    frame(p, o)
                main.wait_stream(side)
            else:
                frame(p, o)
    for s, w in zip(sets, want):
        held.copy_(s)
        graph.replay()
        torch.cuda.synchronize()
        for i, o in enumerate(outs):
            _equal(torch, o, empty if i == 2 else w)


@pytest.mark.parametrize("dims", [(2, 2, 2), (3, 2, 5), (16, 16, 16), (17, 16, 15), (33, 64, 65)])
@pytest.mark.parametrize("offset", [0, 1, 2, 3])
def test_density_is_cleared_at_any_alignment(gpu, dims, offset):
    """Every voxel of the caller's density is cleared, and nothing beside it."""
    hh, torch = gpu
    n = dims[0] * dims[1] * dims[2]
    buf = torch.full((n + 8,), float("nan"), device="cuda")
    far = torch.tensor([[-1e6, 0.0, 0.0, 1.0]], device="cuda")  # reaches no voxel
    hh.hh_splat_density(far, hh.make_grid(dims, 1.0), buf[offset:offset + n])
    got = buf.cpu().numpy()
    assert (got[offset:offset + n] == 0.0).all()
    assert np.isnan(got[:offset]).all() and np.isnan(got[offset + n:]).all()
