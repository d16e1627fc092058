"""The near form of the global search (points just outside the grid, answered from the voxel rows round them) against
the oracle: same neighbours, same squared distances and the same number of global searches, on the dense and the
sparse grid, at every face, edge and corner, from touching distances to where the brick search takes over.  (The near
form serves searches of more than 16,384 points with at most 32 voxels of grid for each.)"""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import assert_nn_equal, gpu_grid, oracle_grid_for, to_np, vicp

pytestmark = pytest.mark.gpu


def _cloud(rng, n, lo, hi):
    p = np.zeros((n, 4), np.float32)
    p[:, :3] = rng.uniform(lo, hi, (n, 3))
    return p


def _round_the_box(rng, lo, hi, gap, n):
    """n points at distances up to `gap` outside random faces, edges and corners of the box."""
    lo, hi = np.asarray(lo, np.float64), np.asarray(hi, np.float64)
    p = rng.uniform(lo, hi, (n, 3))
    side = rng.integers(-1, 2, (n, 3))
    side[(side == 0).all(1), 0] = 1
    d = rng.uniform(0.0, gap, (n, 3)) ** 1.5
    p = np.where(side < 0, lo - d, np.where(side > 0, hi + d, p))
    out = np.zeros((n, 4), np.float32)
    out[:, :3] = p
    return out


def _check(ctx, target, L, src, grid=None):
    """Searches src at the identity pose and compares with the oracle's result on the given (or the fitted) grid."""
    T = torch.eye(4, dtype=torch.float64, device="cuda")
    nn, d2, nf = ctx.correspond(torch.from_numpy(src).cuda(), T)
    assert ctx.sync() == 0
    g, ref = grid
    rnn, rd2, rfb = oracle.correspond(g, ref, target, src, np.eye(4))
    assert int(to_np(nf)[0]) == int(rfb.sum())
    assert np.array_equal(to_np(nn), rnn)
    assert_nn_equal(to_np(nn), to_np(d2), rnn, rd2)


@pytest.mark.parametrize("sparse", [False, True])
@pytest.mark.parametrize("dims", [(1, 1, 1), (5, 1, 7), (33, 9, 4), (40, 70, 65)])
@pytest.mark.parametrize("gap", [1e-6, 0.7, 4.0, 14.0])
def test_points_round_the_grid(dims, gap, sparse):
    """gap in voxels of 0.05: the points nearest to the box reach a few rows, the farthest ones the brick search."""
    v = vicp()
    rng = np.random.default_rng(int(1000 * gap) + sum(dims))
    h, o = 0.05, np.array([-0.4, 0.3, 2.0], np.float32)
    hi = o + h * np.asarray(dims)
    target = _cloud(rng, 3000 if dims[0] > 30 else 90, o + 1e-4, hi - 1e-4)
    src = np.concatenate([_round_the_box(rng, o, hi, gap * h, 17000), _cloud(rng, 200, o, hi)])
    kw = dict(L=6, voxel_size=h, origin=tuple(float(x) for x in o), dims=dims)
    ctx, g = gpu_grid(target, **kw)
    grid = oracle_grid_for(g, target, 6)
    if sparse:
        ctx = v.Context(voxel_size=h, origin=kw["origin"], dims=dims, dilation_layers=6, flags=v.VICP_FLAG_SPARSE_GRID)
        t = torch.from_numpy(target).cuda()
        ctx.build_grid(t)
        ctx.dilate()
    _check(ctx, target, 6, src, grid)


@pytest.mark.parametrize("n_out", [0, 1, 64, 65])
def test_targets_outside_an_explicit_grid(n_out):
    """Target points outside the grid are candidates of every global search, whichever form answers it."""
    rng = np.random.default_rng(n_out)
    o, h, dims = (0.0, 0.0, 0.0), 0.1, (10, 10, 10)
    target = np.concatenate([_cloud(rng, 400, 0.0, 0.999), _round_the_box(rng, [0] * 3, [1] * 3, 0.3, 64)[:n_out],
                             _cloud(rng, 1, 1.01, 1.02)[:min(n_out, 1)]])[:400 + n_out]
    src = _round_the_box(rng, [0] * 3, [1] * 3, 0.4, 17000)
    ctx, g = gpu_grid(np.ascontiguousarray(target), L=4, voxel_size=h, origin=o, dims=dims)
    _check(ctx, target, 4, src, oracle_grid_for(g, target, 4))


def test_equal_and_vanishing_distances():
    """Duplicate target points, queries that coincide with one, and distances whose squares underflow: ties go to the
    smaller index."""
    h = 1.0
    target = np.zeros((40, 4), np.float32)
    target[:, 0] = np.repeat([0.0, 3.0], 20)
    target[20:30, 1] = 1e-25
    src = np.zeros((60, 4), np.float32)
    src[:20, 0] = -1e-30               # outside by less than any square can show
    src[20:40, 0] = -np.float32(2.0) ** -np.arange(20)
    src[40:, 0] = 4.0 + 0.25 * np.arange(20)
    src[40:, 1] = 1e-25
    ctx, g = gpu_grid(target, L=3, voxel_size=h, origin=(0.0, 0.0, 0.0), dims=(4, 1, 1))
    _check(ctx, target, 3, np.tile(src, (300, 1)), oracle_grid_for(g, target, 3))


@pytest.mark.parametrize("offset", [10.0, 300.0, 4000.0])
def test_grids_far_from_the_origin(offset):
    """Coordinates whose rounding is a small or a large part of a voxel."""
    rng = np.random.default_rng(int(offset))
    h, dims = 0.002, (60, 50, 40)
    o = np.array([offset, -offset, 0.25 * offset], np.float32)
    hi = o + h * np.asarray(dims)
    target = _cloud(rng, 2000, o, hi)
    ctx, g = gpu_grid(target, L=6, voxel_size=h, origin=tuple(float(x) for x in o), dims=dims)
    src = np.concatenate([_round_the_box(rng, o, hi, 3 * h, 17000), _cloud(rng, 200, o, hi)])
    _check(ctx, target, 6, src, oracle_grid_for(g, target, 6))


@pytest.mark.parametrize("nz", [80, 81])
@pytest.mark.parametrize("n", [16384, 16385, 17000])
def test_where_the_rows_begin(n, nz):
    """32 voxels a query (80 x 85 x 80 for 17,000) and 16,384 queries: either side of both lines."""
    rng = np.random.default_rng(n + nz)
    h, o, dims = 0.05, np.array([0.1, -0.2, 0.3], np.float32), (80, 85, nz) if n == 17000 else (20, 24, nz)
    hi = o + h * np.asarray(dims)
    target = _cloud(rng, 4000, o, hi)
    src = np.concatenate([_round_the_box(rng, o, hi, 2 * h, n - 1000), _cloud(rng, 500, o, hi),
                          _round_the_box(rng, o - 20 * h, hi + 20 * h, h, 500)])
    rng.shuffle(src)
    ctx, g = gpu_grid(target, L=6, voxel_size=h, origin=tuple(float(x) for x in o), dims=dims)
    _check(ctx, target, 6, src, oracle_grid_for(g, target, 6))
