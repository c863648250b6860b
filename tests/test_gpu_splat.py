"""The splat's box kernels over their smoothing lengths, against the FP64 oracle.

One length at, just inside and just beyond every line of the choice between
box sizes, and the wide kernel beyond the last; ragged grids down to ones
thinner than the support; particles everywhere, on voxel centres and corners,
with supports that end on centres, across the faces, outside, and at
non-finite positions, which add nothing.
"""
import numpy as np
import pytest

import hh_inputs as hi

pytestmark = pytest.mark.gpu

LENGTHS = [0.2, 0.5, 0.8, 1.0, 1.01, 1.5, 1.51, 1.99, 2.01, 2.5, 2.51, 3.0, 3.01, 4.0, 4.01]


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    from paper_2603_02048_gb300 import hh

    return hh, torch


def _particles(dims, h, seed):
    g = np.random.default_rng(seed)
    free = hi.random_particles(400, dims, seed=seed, margin=-2 * h)
    axis = np.concatenate([np.arange(-2, 22) + 0.5, np.arange(-2, 22) * 1.0,
                           np.arange(0, 20) + 0.5 + 2 * h - np.floor(2 * h)])
    edge = np.concatenate([g.choice(axis, size=(200, 3)), g.uniform(0.5, 2.0, (200, 1))], axis=1)
    odd = np.array([[np.nan, 5, 5, 1], [5, np.inf, 5, 1], [5, 5, -np.inf, 1], [1e30, 5, 5, 1],
                    [-4e4, 5, 5, 1]])
    return np.concatenate([free, edge, odd]).astype(np.float32)


@pytest.mark.parametrize("h", LENGTHS)
@pytest.mark.parametrize("dims", [(37, 29, 21), (3, 5, 40)])
def test_splat_over_smoothing_lengths(gpu, oracle_lib, dims, h):
    hh, torch = gpu
    h = float(np.float32(h))
    parts = _particles(dims, h, seed=int(100 * h) + dims[0])
    rho = torch.full((dims[0] * dims[1] * dims[2],), float("nan"), device="cuda")
    hh.hh_splat_density(torch.from_numpy(parts).cuda(), hh.make_grid(dims, h), rho)
    got = rho.cpu().numpy().astype(np.float64).reshape(dims[::-1])
    want = oracle_lib.splat(parts[np.isfinite(parts).all(axis=1)], dims, h)
    # as test_splat_matches_oracle: FP32 kernel values (a distance is off by at most
    # a few 2^-24 of the coordinate, below 64) and FP32 sums in any order
    assert np.abs(got - want).max() <= 1e-5 * want.max() + 1e-30
