"""The one-cluster iterations of small source clouds and the separate kernels give the same bits, so that neither kernel
timing, nor the sparse grid, nor what was called before (a step after a build takes the separate kernels where the grid
before it was built for one step, too) shows in a result.  And which of the two ran: one launch or three."""
import numpy as np
import pytest
import torch

from gpu_util import context, vicp
from paper_2512_04996_gb300 import synth

pytestmark = pytest.mark.gpu


def _clouds(m):
    p = synth.sphere_plane(seed=m + 7, n=max(5000, m))
    s = p.source[np.random.default_rng(m).permutation(p.source.shape[0])[:m]]
    return torch.from_numpy(np.ascontiguousarray(s)).cuda(), torch.from_numpy(p.target).cuda()


@pytest.mark.parametrize("m", [3, 33, 255, 257, 1025, 8192, 8193, 16384, 16385, 24575, 24576, 24577])
def test_paths_agree_bit_for_bit(m):
    v = vicp()
    s, t = _clouds(m)
    rebuild = v.VICP_FLAG_KEEP_GRID | v.VICP_FLAG_REBUILD_EACH_ITER
    res = []
    for flags, timing in ((0, False), (0, True), (v.VICP_FLAG_KEEP_GRID, False), (rebuild, False), (rebuild, True),
                          (v.VICP_FLAG_SPARSE_GRID, False)):
        ctx = context(divisions=64, max_iters=6, eps=1e-9, flags=flags)
        if timing:
            ctx.profile_enable()
        res += [ctx.register(s, t) for _ in range(3)]   # (the later ones replayed as a graph, where one is)
    for r in res:
        assert r[0] == res[0][0] and r[2:] == res[0][2:] and np.array_equal(r[1], res[0][1])


@pytest.mark.parametrize("m", [1000, 8200, 24576])
def test_a_loop_of_builds_and_steps_and_its_launches(m):
    s, t = _clouds(m)
    ctx = context(divisions=64, flags=vicp().VICP_FLAG_KEEP_GRID)
    kept = context(divisions=64, flags=vicp().VICP_FLAG_KEEP_GRID)
    kept.build_grid(t)
    kept.dilate()
    a, b = (torch.eye(4, dtype=torch.float64, device="cuda") for _ in range(2))
    r, q = (torch.zeros(1, dtype=torch.float64, device="cuda") for _ in range(2))
    launches = []
    for _ in range(4):
        ctx.build_grid(t)
        ctx.dilate()
        n0 = ctx.launch_count()
        ctx.step(s, a, r)
        launches.append(ctx.launch_count() - n0)
        kept.step(s, b, q)
        assert ctx.sync() == kept.sync() == 0
        assert torch.equal(a, b) and torch.equal(r, q)
    assert launches[1:] == [3, 3, 3]   # (at the first build nothing is known yet)
    n0 = kept.launch_count()
    for _ in range(3):
        kept.step(s, b, q)
    assert kept.launch_count() - n0 == 3


def test_a_loop_that_fits_its_grids_keeps_the_one_launch():
    """(Nothing overlaps where the host reads every cloud's box, so there is nothing to gain from three.)"""
    s, t = _clouds(1500)
    ctx = context(divisions=64)
    a = torch.eye(4, dtype=torch.float64, device="cuda")
    for _ in range(3):
        ctx.build_grid(t)
        ctx.dilate()
        n0 = ctx.launch_count()
        ctx.step(s, a)
        assert ctx.launch_count() - n0 == 1
    assert ctx.sync() == 0
