"""The brick scan of large grids (more than 65536 brick slots, two launches over tiles of 4096) through what depends on
it: the exact global search, against the oracle, at slot counts just past the limit and at whole and ragged tiles."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import assert_nn_equal, gpu_grid, oracle_grid_for, to_np

pytestmark = pytest.mark.gpu


# dims in voxels; a super-brick is 32 voxels along an axis and holds 64 slots
@pytest.mark.parametrize("supers", [(1024, 1, 1), (1025, 1, 1), (1088, 1, 1), (1089, 1, 1), (33, 8, 9), (1, 1, 2200)])
def test_global_search_over_many_brick_slots(supers):
    rng = np.random.default_rng(sum(supers))
    dims = tuple(32 * k - 25 if k > 1 else 6 for k in supers)
    h = 0.01
    size = h * np.asarray(dims)
    target = np.zeros((3000, 4), np.float32)
    target[:, :3] = rng.uniform(0.0, 0.9999, (3000, 3)) * size
    target[:700, :3] = rng.uniform(0.0, 0.02, (700, 3)) * size           # the first slots
    target[700:1400, :3] = size * 0.9999 - rng.uniform(0.0, 0.02, (700, 3)) * size   # the last ones
    src = np.zeros((1500, 4), np.float32)
    src[:, :3] = rng.uniform(-0.1, 1.1, (1500, 3)) * size
    ctx, g = gpu_grid(target, L=1, voxel_size=h, origin=(0.0, 0.0, 0.0), dims=dims)
    grid, ref = oracle_grid_for(g, target, 1)
    T = torch.eye(4, dtype=torch.float64, device="cuda")
    for again in range(2):   # and rebuilt: the counts return to zero between builds
        nn, d2, nf = ctx.correspond(torch.from_numpy(src).cuda(), T)
        assert ctx.sync() == 0
        rnn, rd2, rfb = oracle.correspond(grid, ref, target, src, np.eye(4))
        assert int(to_np(nf)[0]) == int(rfb.sum()) > 1000
        assert np.array_equal(to_np(nn), rnn)
        assert_nn_equal(to_np(nn), to_np(d2), rnn, rd2)
        ctx.build_grid(g["_target"])
        ctx.dilate(1)
