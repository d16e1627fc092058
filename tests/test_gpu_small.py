"""ICP iterations of a small source cloud by one thread-block cluster (up to 24576 points) against the separate kernels,
which a context with kernel timing enabled runs, and against the oracle.  Same matches, so the sums differ only by
their order: poses within 1e-12 (double-float sums carry about 2^-46), the same iteration counts and statuses."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import context, rot_err
from paper_2512_04996_gb300 import synth

pytestmark = pytest.mark.gpu


def _pair(m, n=5000):
    p = synth.sphere_plane(seed=m, n=max(n, m))
    rng = np.random.default_rng(m)
    src = np.ascontiguousarray(p.source[rng.permutation(p.source.shape[0])[:m]])
    return p, torch.from_numpy(src).cuda(), torch.from_numpy(p.target).cuda(), src


def _close(a, b, tol=1e-12):
    return float(np.abs(np.asarray(a) - np.asarray(b)).max()) <= tol


@pytest.mark.parametrize("m", [1, 2, 3, 31, 32, 33, 127, 128, 129, 255, 257, 1000, 2047, 2049, 8191, 8193, 16384, 16385, 24575, 24576,
                               24577])
def test_step_and_registration_equal_the_separate_kernels(m):
    p, s, t, src = _pair(m)
    out = []
    for timing in (False, True):
        ctx = context(divisions=64, max_iters=6)
        if timing:
            ctx.profile_enable()
        st, T, it, rmse = ctx.register(s, t)
        pose = torch.eye(4, dtype=torch.float64, device="cuda")
        r = torch.zeros(1, dtype=torch.float64, device="cuda")
        ctx.read_stats(reset=True)
        ctx.step(s, pose, r)
        step_st = ctx.sync()
        stats = ctx.read_stats()
        out.append((st, T, it, rmse, step_st, pose.cpu().numpy(), float(r[0]), stats["queries"], stats["fallbacks"]))
    a, b = out
    assert (a[0], a[2], a[4], a[7], a[8]) == (b[0], b[2], b[4], b[7], b[8])
    assert _close(a[1], b[1]) and _close(a[5], b[5]) and _close(a[3], b[3]) and _close(a[6], b[6])
    if m >= 1000:
        grid = oracle.fit_grid(p.target, 0.0, 64)
        _, R, rit, _ = oracle.register(grid, 10, p.target, src, np.eye(4), max_iters=6, eps=0.0)
        assert rit == a[2] and rot_err(a[1], R) <= 1e-5 and np.linalg.norm(a[1][:3, 3] - R[:3, 3]) <= 2e-5


@pytest.mark.parametrize("rebuild", [False, True])
@pytest.mark.parametrize("eps", [1e-3, 1e-5])
def test_stopping_rule(eps, rebuild):
    """The RMSE test across launches of one iteration (the grid rebuilt) and within one launch of all of them."""
    v = __import__("paper_2512_04996_gb300.vicp", fromlist=["x"])
    p, s, t, src = _pair(4096, 4096)
    flags = v.VICP_FLAG_KEEP_GRID | (v.VICP_FLAG_REBUILD_EACH_ITER if rebuild else 0)
    res = []
    for timing in (False, True):
        ctx = context(divisions=64, max_iters=40, eps=eps, flags=flags)
        if timing:
            ctx.profile_enable()
        res.append([ctx.register(s, t) for _ in range(3)])   # (the later ones replayed as a graph)
    for x, y in zip(*res):
        assert x[0] == y[0] == 0 and x[2] == y[2] < 40 and _close(x[1], y[1]) and _close(x[3], y[3])
    assert all(np.array_equal(r[1], res[0][0][1]) for r in res[0])


def test_dense_segments_and_far_queries():
    """A dense target (hundreds of points a voxel) and sources far from it, outside the grid and not finite."""
    rng = np.random.default_rng(3)
    target = np.zeros((30000, 4), np.float32)
    target[:, :3] = rng.uniform(-1, 1, (30000, 3)) * [1.0, 1.0, 0.02]
    src = np.zeros((3000, 4), np.float32)
    src[:, :3] = rng.uniform(-1, 1, (3000, 3)) * [1.0, 1.0, 0.02] + [0.01, 0.02, 0.01]
    src[2500:, :3] = rng.uniform(-3, 3, (500, 3))
    s, t = torch.from_numpy(src).cuda(), torch.from_numpy(target).cuda()
    res = []
    for timing in (False, True):
        ctx = context(voxel_size=0.2, L=3, max_iters=4)
        if timing:
            ctx.profile_enable()
        res.append(ctx.register(s, t))
    a, b = res
    assert a[0] == b[0] == 0 and a[2] == b[2] == 4 and _close(a[1], b[1]) and _close(a[3], b[3])
