"""The calls of this framework whose speed is measured, with their inputs.

A case is one call (or one short run of calls) that a renderer built on the
library makes each frame or each request, through the public binding
`paper_2603_02048_gb300.hh`:

  splat     hh_splat_density: particles to density
  field     hh_build_index_field_noalloc: particles to the caller's volume
  trace     hh_trace of one view on a volume that is already there
  frame     hh_volume_rebuild + hh_trace (one view) or hh_batch_launch_graph
            (several): a simulation frame from particles to images
  pipeline  hh_pipeline_submit / hh_pipeline_wait: host particles in, host
            display images out, several frames in flight
  serve     hh_serve_submit / hh_serve_wait: several requests at once against
            a resident volume

Sizes are those of the tests, of the benchmark and of its inputs (64^3 to
512^3 voxels, 128x128 to 3840x2160 pixels, 1 to 32 views), or ragged ones in
the same range. Everything is drawn on the GPU from the seed. `exact` restates
the method in 64-bit torch, without the library.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_2603_02048_gb300 import hh

K_GD = float(np.float32(2.26e-4))
# uneven views of a batch, and of the render server's requests
BATCH_RESOLUTIONS = ((256, 256), (640, 480), (1280, 720), (1920, 1080))
SERVE_RESOLUTIONS = ((320, 240), (1280, 720), (1920, 1080), (3840, 2160))


def _case(name, kind, dims, **more):
    c = {"kind": kind, "nx": dims[0], "ny": dims[1], "nz": dims[2], "scene": "plume", "n": 0,
         "h": 2.0, "storage": "fp32", "stepper": "euler", "theta": 3e-5, "step": 2.0, "views": 1,
         "w": 0, "px": 0, "mix": False, "out": "rgb", "planes": 0, "tile_order": 0,
         "tile_group": 0, "repeat": 1}
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the density of the headline frame's particles, for a caller that
        # only wants the splat (a fluid solver's own grid)
        _case("splat 256^3", "splat", (256, 256, 256), n=262144),
        # a wider smoothing length on a ragged grid, particles everywhere up
        # to the faces
        _case("splat h=3 ragged", "splat", (161, 118, 97), scene="uniform", n=60011, h=3.0),
        # a host that owns all device memory: the largest cube that the
        # allocation-free build takes
        _case("field noalloc 128^3", "field", (128, 128, 128), n=65536),
        # the smallest call: a preview of a given index volume, RK4 at half a
        # voxel, every output
        _case("trace 64^3 rk4 128x128", "trace", (64, 64, 64), scene="dn", stepper="rk4",
              theta=0.0, step=0.5, w=128, px=128, out="all"),
        # a turbulence volume without any empty space, one 720p view with
        # every output (angle-of-arrival statistics), the step varying
        _case("trace turbulence 720p", "trace", (192, 160, 224), scene="turbulence", theta=1e-5,
              w=1280, px=720, out="all"),
        # odd sizes throughout: FP16 storage, adaptive RK4, two boards behind
        # the plume
        _case("trace fp16 rk4 ragged", "trace", (93, 118, 77), scene="blobs", storage="fp16",
              stepper="rk4", w=641, px=363, out="both", planes=2),
        # one 4K view, the benchmark's calibrated tolerance
        _case("trace fp16 4k", "trace", (384, 384, 384), scene="blobs", storage="fp16", w=3840,
              px=2160),
        # the headline frame (whole frames run at the paper's tolerance, where
        # every ray is well conditioned: the splat's atomic sums differ in the
        # last bits from run to run)
        _case("frame 256^3 1080p", "frame", (256, 256, 256), n=262144, theta=3e-3, w=1920, px=1080),
        # the eight-view arc on FP16 storage, one graph-replayed launch
        _case("frame 256^3 fp16 8 views", "frame", (256, 256, 256), n=262144, storage="fp16",
              theta=3e-3, views=8, w=1280, px=720, tile_order=1),
        # the largest frame: 32 uneven views of a 512^3 volume
        _case("frame 512^3 fp16 32 views", "frame", (512, 512, 512), n=2097152, storage="fp16",
              theta=3e-3, views=32, mix=True, tile_order=1, tile_group=1),
        # the real-time loop, host buffers on both ends, a tolerance at which
        # the step follows the plume's fine structure
        _case("pipeline 256^3 1080p", "pipeline", (256, 256, 256), n=262144, theta=1e-5, w=1920,
              px=1080, out="rgb8", repeat=4),
        # a burst of requests of uneven size to the render server
        _case("serve 384^3 fp16 burst", "serve", (384, 384, 384), n=1048576, storage="fp16",
              theta=3e-3, views=3, mix=True, repeat=6),
    ]


def draw(rng):
    def between(lo, hi):  # over the logarithm
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def grid(lo, hi):
        n = between(lo, hi)
        return tuple(max(8, int(n * rng.uniform(0.7, 1.3))) if rng.random() < 0.5 else n
                     for _ in range(3))

    def density(dims, rate):  # particles at `rate` to the headline frame's density
        return max(64, int(262144 * rate * dims[0] * dims[1] * dims[2] / 256.0**3))

    kind = rng.choice(("splat", "field", "trace", "trace", "frame", "frame", "pipeline", "serve"))
    if kind == "splat":
        d = grid(48, 320)
        return _case(None, kind, d, scene=rng.choice(("plume", "uniform")),
                     n=density(d, rng.uniform(0.3, 3.0)),
                     h=rng.choice((1.0, 1.5, 2.0, 2.0, 2.5, 3.0)))
    if kind == "field":
        d = tuple(rng.randint(24, 126) for _ in range(3))
        return _case(None, kind, d, n=density(d, rng.uniform(0.5, 3.0)))
    storage = rng.choice(("fp32", "fp16"))
    theta = rng.choice((0.0, 1e-5, 3e-5, 3e-3) if kind == "trace" else (0.0, 3e-3))
    step = rng.choice((0.5, 1.0, 2.0)) if theta == 0.0 else 2.0
    w, px = between(100, 2000), between(80, 1200)
    if kind == "trace":
        return _case(None, kind, grid(40, 320), scene=rng.choice(("dn", "turbulence", "blobs")),
                     storage=storage, theta=theta, step=step, w=w, px=px,
                     stepper=rng.choice(("euler", "euler", "rk4")),
                     out=rng.choice(("rgb", "rgb8", "all")), planes=rng.choice((0, 0, 1, 2)))
    d = grid(64, 320)
    n = density(d, rng.uniform(0.3, 2.0))
    if kind == "frame":
        v = rng.choice((1, 2, 4, 8, 12))
        return _case(None, kind, d, n=n, storage=storage, theta=theta, step=step, views=v, w=w,
                     px=px, mix=v > 1 and rng.random() < 0.5, tile_order=rng.randint(0, 1),
                     tile_group=rng.randint(0, 1))
    if kind == "pipeline":
        return _case(None, kind, grid(128, 280), n=between(100000, 400000), storage=storage,
                     theta=1e-5, views=rng.choice((1, 1, 2)), w=between(1280, 2000),
                     px=between(720, 1200), out="rgb8", repeat=rng.randint(2, 5))
    return _case(None, kind, d, n=n, storage="fp16", theta=theta, step=step,
                 views=rng.randint(1, 4), mix=True, repeat=rng.randint(1, 6))


# --------------------------------------------------------------------------- #
# inputs
# --------------------------------------------------------------------------- #
def _dims(case):
    return case["nx"], case["ny"], case["nz"]


def _generator(seed, part):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 16 + part)
    return g


def _particles(case, seed, frame=0):
    """(n, 4) float32 {x, y, z, m}: a hot plume (Gaussian, rising, clear of the
    faces by one support) or a uniform cloud up to the faces."""
    g = _generator(seed, 1 + frame)
    n, dims, h = case["n"], _dims(case), case["h"]
    size = torch.tensor(dims, device="cuda", dtype=torch.float32)
    if case["scene"] == "uniform":
        pos = torch.rand((n, 3), generator=g, device="cuda") * size
        m = torch.rand((n, 1), generator=g, device="cuda") * 1.5 + 0.5
        return torch.cat([pos, m], 1).contiguous()
    sigma = 0.15 * size
    mean = 0.5 * size + torch.tensor([0.0, 0.0, 0.075], device="cuda") * size
    pos = torch.empty((0, 3), device="cuda")
    while pos.shape[0] < n:
        new = torch.randn((n + 1024, 3), generator=g, device="cuda") * sigma + mean
        keep = ((new >= 2 * h) & (new <= size - 2 * h)).all(1)
        pos = torch.cat([pos, new[keep]])
    out = torch.empty((n, 4), device="cuda")
    out[:, :3] = pos[:n]
    out[:, 3] = 1.2 * (2 * math.pi) ** 1.5 * 0.15**3 * dims[0] * dims[1] * dims[2] / n
    return out


def _dn(case, seed):
    """A given dn grid (nz, ny, nx): the smooth 64^3 scene's kind ("dn"), the
    same cut off at 2 % of its peak, so that most of the box is exactly empty
    ("blobs"), or homogeneous turbulence ("turbulence", no empty space)."""
    g = _generator(seed, 2)
    nx, ny, nz = _dims(case)
    if case["scene"] == "turbulence":
        noise = torch.randn((nz, ny, nx), generator=g, device="cuda")
        k2 = (torch.fft.fftfreq(nz, device="cuda")[:, None, None] ** 2
              + torch.fft.fftfreq(ny, device="cuda")[None, :, None] ** 2
              + torch.fft.rfftfreq(nx, device="cuda")[None, None, :] ** 2)
        f = torch.fft.irfftn(torch.fft.rfftn(noise) * torch.exp(-2 * (math.pi * 2.0) ** 2 * k2),
                             s=(nz, ny, nx))
        return (f * (1e-5 / f.std())).contiguous()
    r = torch.rand((8, 5), generator=g, device="cuda").cpu().tolist()
    size = (nx + ny + nz) / 3.0 / 64.0
    ax = [torch.arange(m, device="cuda", dtype=torch.float32) + 0.5 for m in (nx, ny, nz)]

    def bump(c, s):
        ex, ey, ez = (torch.exp(-((a - p) ** 2) / (2 * s * s)) for a, p in zip(ax, c))
        return ez[:, None, None] * ey[None, :, None] * ex[None, None, :]

    dn = -3e-5 * bump((nx / 2, ny / 2, nz / 2), 12.0 * size)
    for a, s, x, y, z in r:
        c = [(0.125 + 0.75 * t) * m for t, m in zip((x, y, z), (nx, ny, nz))]
        dn += (4e-5 * a - 2e-5) * bump(c, (3.0 + 5.0 * s) * size)
    if case["scene"] == "blobs":
        dn[dn.abs() < 0.02 * dn.abs().max()] = 0.0
    return dn.contiguous()


def _background(seed):
    """RGB8 equirect map: 16 x 16 checker with noise."""
    g = _generator(seed, 3)
    i = torch.arange(512, device="cuda") * 16 // 512
    base = torch.where((i[:, None] + i[None, :]) % 2 == 0, 0.2, 0.8)
    img = base[:, :, None] + torch.rand((512, 512, 3), generator=g, device="cuda") * 0.2 - 0.1
    return (img.clamp(0, 1) * 255).round().to(torch.uint8).contiguous()


def _planes(case, bg):
    """Boards behind the volume (seen from -x), at different depths."""
    nx, ny, nz = _dims(case)
    out = []
    for k in range(case["planes"]):
        depth = 0.5 + k
        half = 0.6 * nx * (1.0 + depth)
        out.append({"origin": [nx + depth * nx, ny / 2 - half, nz / 2 - half],
                    "u": [0.0, 2 * half, 0.0], "v": [0.0, 0.0, 2 * half],
                    "tex": bg[64 * k:64 * k + 256, :256].contiguous()})
    return out


def _orbit(dims, azimuth, elevation, w, px):
    c = [d / 2.0 for d in dims]
    dist = 1.5 * max(dims)
    az, el = math.radians(azimuth), math.radians(elevation)
    d = (math.cos(az) * math.cos(el), math.sin(az) * math.cos(el), math.sin(el))
    return {"eye": [c[k] - dist * d[k] for k in range(3)], "look_at": c, "up": [0.0, 0.0, 1.0],
            "vfov_deg": 60.0, "width": int(w), "height": int(px)}


def _cameras(case, seed, resolutions=BATCH_RESOLUTIONS, request=0):
    """One view near the -x side; several of one size on a 90 degree arc; or
    an uneven mix all around."""
    r = np.random.Generator(np.random.PCG64([int(seed), 4, request]))
    v, dims = case["views"], _dims(case)
    if case["mix"]:
        # resolutions in turn, so that every seed has the same number of rays
        sizes = [resolutions[(k + request) % len(resolutions)] for k in range(v)]
        return [_orbit(dims, r.uniform(0, 360), r.uniform(-30, 30), w, px) for w, px in sizes]
    turn = r.uniform(-5, 5)
    az = [0.0] if v == 1 else [-45 + 90 * k / (v - 1) for k in range(v)]
    return [_orbit(dims, a + turn, turn / 2, case["w"], case["px"]) for a in az]


def _params(case):
    least = case["step"] if case["theta"] == 0.0 else 0.125
    diag = math.sqrt(sum(d * d for d in _dims(case)))
    return {"stepper": case["stepper"], "adaptive": case["theta"] > 0.0, "h_fixed": case["step"],
            "h_min": 0.125, "h_max": 2.0, "theta_max": case["theta"], "eps": 1e-6,
            "max_steps": int(math.ceil(3 * diag / least))}


def _outputs(case, cam):
    n = cam["width"] * cam["height"]
    want = {"rgb": ("rgb",), "rgb8": ("rgb8",), "both": ("rgb", "rgb8"),
            "all": ("rgb", "exit_pos", "exit_dir", "steps", "flags")}[case["out"]]
    kinds = {"rgb8": torch.uint8, "steps": torch.int32, "flags": torch.int32}
    return {k: torch.zeros(n if k in ("steps", "flags") else 3 * n, device="cuda",
                           dtype=kinds.get(k, torch.float32)) for k in want}


class _Server:
    """The process's render server, and one put volume for as long as its
    state lives."""

    server = None
    ids = itertools.count()

    def __init__(self, vol):
        if _Server.server is None:
            _Server.server = hh.hh_serve_create(2 << 30, 16)
        self.frame = next(_Server.ids)
        hh.hh_serve_put_volume(_Server.server, self.frame, vol)

    def __del__(self):
        try:
            hh.hh_serve_remove_volume(_Server.server, self.frame)
        except Exception:  # the interpreter is going down
            pass


def prepare(case, seed):
    kind, dims = case["kind"], _dims(case)
    grid = hh.make_grid(dims, case["h"], case["storage"])
    s = {"case": case, "grid": grid}
    if kind in ("splat", "field"):
        s["parts"] = _particles(case, seed)
        s["out"] = torch.empty(dims[0] * dims[1] * dims[2] * (1 if kind == "splat" else 4),
                               device="cuda")
        torch.cuda.synchronize()
        return s
    s["bg_t"] = _background(seed)
    s["planes"] = _planes(case, s["bg_t"])
    s["bg"] = hh.make_background(s["bg_t"], s["planes"])
    s["params"] = hh.make_params(_params(case))
    if kind == "serve":
        parts = _particles(case, seed)
        s["vol"] = hh.hh_build_index_field(parts, grid, K_GD)
        torch.cuda.synchronize()
        s["put"] = _Server(s["vol"])
        dicts = [_cameras(case, seed, SERVE_RESOLUTIONS, q) for q in range(case["repeat"])]
        s["sizes"] = [[(c["width"], c["height"]) for c in cams] for cams in dicts]
        s["cams"] = [[hh.make_camera(c) for c in cams] for cams in dicts]
        return s
    cams = _cameras(case, seed)
    s["cams"] = [hh.make_camera(c) for c in cams]
    if kind == "pipeline":
        s["host"] = [_particles(case, seed, f).cpu().pin_memory() for f in range(case["repeat"])]
        s["images"] = [[torch.zeros(3 * c["width"] * c["height"], dtype=torch.uint8).pin_memory()
                        for c in cams] for _ in range(case["repeat"])]
        s["pipe"] = hh.hh_pipeline_create(grid, K_GD, case["n"], s["cams"], s["params"], s["bg"])
        return s
    s["outs"] = [_outputs(case, c) for c in cams]
    if kind == "trace":
        dn = _dn(case, seed)
        s["vol"] = hh.hh_volume_from_dn(dn.view(-1), grid)
        torch.cuda.synchronize()
        return s
    s["parts"] = _particles(case, seed)
    s["vol"] = hh.hh_build_index_field(s["parts"], grid, K_GD)
    torch.cuda.synchronize()
    if case["views"] > 1:
        s["stream"] = torch.cuda.Stream()
        s["batch"] = hh.hh_batch_create(s["vol"], s["cams"], s["params"], s["bg"], s["outs"])
        hh.hh_batch_set_config(s["batch"], 128, 0, 32, 4 if case["mix"] else 8,
                               case["tile_order"], case["tile_group"])
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "splat":
        hh.hh_splat_density(s["parts"], s["grid"], s["out"])
        return s["out"]
    if kind == "field":
        hh.hh_build_index_field_noalloc(s["parts"], s["grid"], K_GD, s["out"])
        return s["out"]
    if kind == "trace":
        hh.hh_trace(s["vol"], s["cams"], s["params"], s["bg"], s["outs"])
        return s["outs"]
    if kind == "frame":
        stream = s.get("stream")
        hh.hh_volume_rebuild(s["vol"], s["parts"], K_GD, stream)
        if stream is None:
            hh.hh_trace(s["vol"], s["cams"], s["params"], s["bg"], s["outs"])
        else:
            hh.hh_batch_launch_graph(s["batch"], stream)
        return s["outs"]
    if kind == "pipeline":
        for parts, images in zip(s["host"], s["images"]):
            frame = hh.hh_pipeline_submit(s["pipe"], parts, images)
        hh.hh_pipeline_wait(s["pipe"], frame - 1)
        hh.hh_pipeline_wait(s["pipe"], frame)
        return s["images"]
    server, out = _Server.server, []
    tickets = [hh.hh_serve_submit(server, s["put"].frame, cams, s["params"], s["bg"],
                                  hh.HH_OUT_RGB) for cams in s["cams"]]
    for t, sizes in zip(tickets, s["sizes"]):
        hh.hh_serve_wait(server, t, 20000)
        out.append([hh.hh_serve_view(server, t, v, w, px) for v, (w, px) in enumerate(sizes)])
        hh.hh_serve_release(server, t)
    return out


# --------------------------------------------------------------------------- #
# what a pass cannot do without
# --------------------------------------------------------------------------- #
def work(case):
    """Bytes: particles read, the rebuilt volume or density written, a marched
    volume read once per pass, images written. Flops: 14 per voxel of a
    particle's support, 8 per voxel of the field, 158 per march step (four
    times that for RK4), a ray that enters the box taking half the mean axis
    over its longest step."""
    nx, ny, nz = _dims(case)
    kind, voxels, n = case["kind"], case["nx"] * case["ny"] * case["nz"], case["n"]
    support = 4.0 / 3.0 * math.pi * (2 * case["h"]) ** 3
    store = 16 if case["storage"] == "fp32" else 8
    if kind == "splat":
        return {"bytes": 16 * n + 4 * voxels, "flops": 14 * support * n}
    if kind == "field":
        return {"bytes": 16 * n + 16 * voxels, "flops": 14 * support * n + 8 * voxels}
    views = case["views"]
    if case["mix"]:
        sizes = SERVE_RESOLUTIONS if kind == "serve" else BATCH_RESOLUTIONS
        per = case["repeat"] if kind == "serve" else 1
        pixels = sum(w * px for q in range(per) for w, px in
                     (sizes[(k + q) % len(sizes)] for k in range(views)))
    else:
        pixels = views * case["w"] * case["px"]
    pixel = {"rgb": 12, "rgb8": 3, "both": 15, "all": 44}[case["out"]]
    steps = 0.5 * (nx + ny + nz) / 3.0 / case["step"]
    march = pixels * 0.45 * steps * 158 * (4 if case["stepper"] == "rk4" else 1)
    out = {"bytes": pixels * pixel + store * voxels, "flops": march}
    if kind in ("frame", "pipeline"):
        out["bytes"] += 16 * n + store * voxels
        out["flops"] += 14 * support * n + 8 * voxels
        if kind == "pipeline":
            out = {k: v * case["repeat"] for k, v in out.items()}
    return out


# --------------------------------------------------------------------------- #
# the method in 64 bits
# --------------------------------------------------------------------------- #
def _splat64(parts, dims, h):
    """rho at the voxel centres: the M4 cubic spline of support 2h, in float64."""
    nx, ny, nz = dims
    h = float(np.float32(h))
    rho = torch.zeros(nx * ny * nz, dtype=torch.float64, device="cuda")
    slots = torch.arange(int(math.ceil(4 * h)) + 1, device="cuda")
    size = torch.tensor(dims, device="cuda")
    norm = 1.0 / (math.pi * h**3)
    for p in parts.double().split(max(1, 2**25 // len(slots) ** 3)):
        x = p[:, :3]
        i = torch.floor(x - 2 * h - 0.5).long()[:, :, None] + slots  # (c, 3, s)
        d2 = ((i + 0.5) - x[:, :, None]) ** 2
        ok = (i >= 0) & (i < size[None, :, None])
        q = torch.sqrt(d2[:, 2, :, None, None] + d2[:, 1, None, :, None]
                       + d2[:, 0, None, None, :]) / h
        w = 2 * (1 - q / 2).clamp_min(0) ** 3 - (1 - q).clamp_min(0) ** 3
        keep = (ok[:, 2, :, None, None] & ok[:, 1, None, :, None] & ok[:, 0, None, None, :]
                & (q < 2))
        at = (i[:, 2, :, None, None] * ny + i[:, 1, None, :, None]) * nx + i[:, 0, None, None, :]
        w = w * (p[:, 3] * norm)[:, None, None, None]
        rho.index_add_(0, at[keep], w[keep])
    return rho.view(nz, ny, nx)


def _field64(rho, k):
    """{dn, grad dn} per voxel: central differences, one-sided at the faces."""
    dn = rho.double() * k
    out = torch.empty((*dn.shape, 4), dtype=torch.float64, device="cuda")
    out[..., 0] = dn
    for channel, axis in ((1, 2), (2, 1), (3, 0)):
        out[..., channel] = torch.gradient(dn, dim=axis)[0]
    return out


def _sample64(vol, p):
    """Trilinear sample at positions p, clamped to the voxel centres."""
    nz, ny, nx = vol.shape[:3]
    flat, out = vol.view(-1, 4), 0.0
    cell = []
    for a, n in enumerate((nx, ny, nz)):
        u = (p[:, a] - 0.5).clamp(0, n - 1)
        i = u.floor().clamp_max(n - 2).long()
        cell.append((i, u - i))
    (ix, fx), (iy, fy), (iz, fz) = cell
    for k in (0, 1):
        for j in (0, 1):
            row = ((iz + k) * ny + iy + j) * nx + ix
            w = (fz if k else 1 - fz) * (fy if j else 1 - fy)
            out = out + (w * (1 - fx))[:, None] * flat[row] + (w * fx)[:, None] * flat[row + 1]
    return out


def _bilinear64(tex, s, t, wrap):
    """Bilinear RGB8 lookup at texel coordinates; clamped, or wrapping in s."""
    height, width = tex.shape[:2]
    t = t.clamp(0, height - 1)
    if not wrap:
        s = s.clamp(0, width - 1)
    i0, j0 = s.floor(), t.floor().clamp_max(height - 2)
    if not wrap:
        i0 = i0.clamp_max(width - 2)
    fs, ft = (s - i0)[:, None], (t - j0)[:, None]
    i0, j0 = i0.long(), j0.long()
    i1 = (i0 + 1) % width if wrap else i0 + 1
    i0 = i0 % width
    x = tex.double()
    top = x[j0, i0] * (1 - fs) + x[j0, i1] * fs
    low = x[j0 + 1, i0] * (1 - fs) + x[j0 + 1, i1] * fs
    return (top * (1 - ft) + low * ft) / 255.0


def _scene64(p, d, bg, planes):
    """What the straight ray p + t d sees: the nearest board, else the map."""
    height, width = bg.shape[:2]
    phi, theta = torch.atan2(d[:, 1], d[:, 0]), torch.atan2(d[:, :2].norm(dim=1), d[:, 2])
    rgb = _bilinear64(bg, (phi / (2 * math.pi) + 0.5) * width - 0.5, theta / math.pi * height - 0.5,
                      True)
    near = torch.full_like(phi, math.inf)
    for pl in planes:
        o, u, v = (torch.tensor(np.float32(pl[k]), device="cuda").double()
                   for k in ("origin", "u", "v"))
        normal = torch.linalg.cross(u, v)
        t = ((o - p) @ normal) / (d @ normal)
        r = p + t[:, None] * d - o
        a, b = r @ u / (u @ u), r @ v / (v @ v)
        hit = (t > 0) & (t < near) & (a >= 0) & (a <= 1) & (b >= 0) & (b <= 1)
        th, tw = pl["tex"].shape[:2]
        colour = _bilinear64(pl["tex"], a[hit] * tw - 0.5, b[hit] * th - 0.5, False)
        rgb[hit] = colour
        near = torch.where(hit, t, near)
    return rgb


def _rays64(cam):
    cam = {k: np.float32(v).astype(np.float64) if isinstance(v, list) else v
           for k, v in cam.items()}
    f = cam["look_at"] - cam["eye"]
    f /= np.linalg.norm(f)
    r = np.cross(f, cam["up"])
    r /= np.linalg.norm(r)
    f, r, u = (torch.tensor(x, device="cuda") for x in (f, r, np.cross(r, f)))
    width, height = cam["width"], cam["height"]
    t = math.tan(0.5 * math.radians(cam["vfov_deg"]))
    a = (2 * (torch.arange(width, device="cuda").double() + 0.5) / width - 1) * t * width / height
    b = (1 - 2 * (torch.arange(height, device="cuda").double() + 0.5) / height) * t
    d = f + a[None, :, None] * r + b[:, None, None] * u
    d = (d / d.norm(dim=2, keepdim=True)).view(-1, 3)
    return torch.tensor(cam["eye"], device="cuda").expand_as(d), d


def _march64(vol, cams, params, bg, planes):
    """exit_pos, exit_dir and rgb of every ray of the views."""
    P = {k: float(np.float32(v)) if isinstance(v, float) else v for k, v in params.items()}
    nz, ny, nx = vol.shape[:3]
    box = torch.tensor([nx, ny, nz], device="cuda").double()
    o, w = (torch.cat(x) for x in zip(*(_rays64(c) for c in cams)))
    t1, t2 = (0 - o) / w, (box - o) / w
    t_in = torch.minimum(t1, t2).amax(1).clamp_min(0)
    hit = torch.maximum(t1, t2).amin(1) >= t_in
    pos, dirs = o.clone(), w
    live = hit.nonzero()[:, 0]
    c, w = o[live] + t_in[live, None] * w[live], w[live]
    c = torch.minimum(c.clamp_min(0), box)

    def rate(p, d):
        s = _sample64(vol, p)
        n, g = 1 + s[:, 0], s[:, 1:]
        return n, g - (d * g).sum(1, keepdim=True) * d

    for _ in range(P["max_steps"]):
        if not live.numel():
            break
        n, g = rate(c, w)
        if P["adaptive"]:
            ds = (n * P["theta_max"] / (g.norm(dim=1) + P["eps"])).clamp(P["h_min"], P["h_max"])
        else:
            ds = torch.full_like(n, P["h_fixed"])
        ds = ds[:, None]
        if P["stepper"] == "euler":
            w = w + ds / n[:, None] * g
            w = w / w.norm(dim=1, keepdim=True)
            step = ds * w
        else:
            k1, w1 = g / n[:, None], w
            w2 = w + ds / 2 * k1
            n, g = rate(c + ds / 2 * w1, w2)
            k2, w3 = g / n[:, None], w + ds / 2 * (g / n[:, None])
            n, g = rate(c + ds / 2 * w2, w3)
            k3, w4 = g / n[:, None], w + ds * (g / n[:, None])
            n, g = rate(c + ds * w3, w4)
            step = ds / 6 * (w1 + 2 * (w2 + w3) + w4)
            w = w + ds / 6 * (k1 + 2 * (k2 + k3) + g / n[:, None])
            w = w / w.norm(dim=1, keepdim=True)
        to = c + step
        out = ((to < 0) | (to > box)).any(1)
        if out.any():
            s, p = step[out], c[out]
            face = torch.where(s > 0, (box - p) / s, torch.where(s < 0, -p / s, math.inf))
            pos[live[out]] = p + face.amin(1).clamp(0, 1)[:, None] * s
            dirs[live[out]] = w[out]
            live, to, w = live[~out], to[~out], w[~out]
        c = to
    pos[live], dirs[live] = c, w
    rgb = torch.cat([_scene64(p, d, bg, planes) for p, d in zip(pos.split(2**21),
                                                                dirs.split(2**21))])
    return {"rgb": rgb, "exit_pos": pos, "exit_dir": dirs}


def exact(case, seed):
    """The float outputs in 64 bits. Stored halves are not restated: an FP16
    volume's images stand against the unrounded volume's. Display bytes, step
    counts and flags have no such value."""
    kind, dims = case["kind"], _dims(case)
    if case["out"] == "rgb8":
        return None
    if kind != "trace":
        rho = _splat64(_particles(case, seed), dims, case["h"])
        if kind == "splat":
            return rho.view(-1)
        vol = _field64(rho, K_GD)
        del rho
        if kind == "field":
            return vol.view(-1)
    else:
        vol = _field64(_dn(case, seed), 1.0)
    bg = _background(seed)
    if kind == "serve":
        return [_images64(case, vol, _cameras(case, seed, SERVE_RESOLUTIONS, q), bg)
                for q in range(case["repeat"])]
    return _images64(case, vol, _cameras(case, seed), bg)


def _images64(case, vol, cams, bg):
    out, planes = [], _planes(case, bg)
    for few in (cams[k:k + 8] for k in range(0, len(cams), 8)):
        got = _march64(vol, few, _params(case), bg, planes)
        sizes = [c["width"] * c["height"] for c in few]
        parts = {k: v.split(sizes) for k, v in got.items()}
        for k, cam in enumerate(few):
            o = {name: None for name in _outputs(case, {"width": 1, "height": 1})}
            out.append({**o, **{n: parts[n][k].reshape(-1) for n in parts if n in o}})
    return out
