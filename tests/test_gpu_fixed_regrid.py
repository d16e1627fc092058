"""The fixed-capacity store after a build of another grid: its slots are of the voxels it was built on, so a search with
the labels of a grid of other dimensions is refused, and served again after a new vicp_fixed_build."""
import pytest
import torch

from gpu_util import vicp
from paper_2512_04996_gb300 import synth

pytestmark = pytest.mark.gpu


def test_search_after_a_build_of_another_grid():
    v = vicp()
    p = synth.sphere_plane(seed=11, n=3000)
    s, t = torch.from_numpy(p.source).cuda(), torch.from_numpy(p.target).cuda()
    large = t * 3.0
    pose = torch.eye(4, dtype=torch.float64, device="cuda")
    ctx = v.Context(v.default_params(voxel_size=0.1, dilation_layers=10))
    ctx.build_grid(t)
    ctx.dilate()
    ctx.fixed_build(t, 3000)
    ref = ctx.correspond(s, pose)
    ctx.build_grid(t)   # the same dimensions: served
    ctx.dilate()
    assert torch.equal(ctx.fixed_correspond(s, pose)[0], ref[0])
    ctx.build_grid(large)
    ctx.dilate()
    with pytest.raises(v.VicpError) as e:
        ctx.fixed_correspond(s, pose)
    assert e.value.status == v.VICP_ERR_STATE
    ctx.fixed_build(large, 3000)
    assert torch.equal(ctx.fixed_correspond(s, pose)[0], ctx.correspond(s, pose)[0])
    assert ctx.sync() == 0
