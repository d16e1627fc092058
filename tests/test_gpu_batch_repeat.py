"""A batch built and registered again gives the same bits: the order of a voxel's points in the store varies from build
to build, and nothing that it decides (the seed of a query outside the grid, where the root voxel holds more points
than are looked at for it) may show in the sums.  Dense voxels, sources half outside the targets' boxes."""
import numpy as np
import pytest
import torch

from gpu_util import vicp
from paper_2512_04996_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("divisions", [24, 48])
def test_registrations_after_builds_of_the_same_clouds(divisions, fp64):
    v = vicp()
    ps = [synth.sphere_plane(seed=90 + k, n=24000 + 511 * k, max_deg=3.0, max_trans=0.02) for k in range(6)]
    tgt = torch.from_numpy(np.concatenate([p.target for p in ps])).cuda()
    src = torch.from_numpy(np.concatenate([p.source for p in ps])).cuda()
    n = np.array([p.target.shape[0] for p in ps], np.int32)
    b = v.Batch(dilation_layers=10, max_iters=12, flags=v.VICP_BATCH_FLAG_FP64 if fp64 else 0)
    first = None
    for _ in range(6):
        b.build(tgt, n, None, np.full(6, divisions, np.int32))
        r = b.register(src, n)
        assert r[0] == 0
        first = first or r
        assert all(np.array_equal(x, y) for x, y in zip(r[1:], first[1:]))
