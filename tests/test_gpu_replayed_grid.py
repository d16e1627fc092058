"""The grid that a replayed registration leaves behind: after a build of another cloud, or with new contents at the
target's address, searches, steps, views and builds that follow a replay see the replayed call's grid, as they do after
a registration launched directly."""
import numpy as np
import pytest
import torch

from gpu_util import to_np, vicp
from paper_2512_04996_gb300 import synth

pytestmark = pytest.mark.gpu


def _cloud(seed, n):
    p = synth.sphere_plane(seed=seed, n=n)
    return torch.from_numpy(p.source).cuda(), torch.from_numpy(p.target).cuda()


@pytest.mark.parametrize("host", [False, True])
@pytest.mark.parametrize("iters", [1, 4])
@pytest.mark.parametrize("n", [4000, 30000])
def test_after_a_build_of_another_cloud(n, iters, host):
    v = vicp()
    kw = dict(grid_divisions=32, dilation_layers=10, max_iters=iters, rmse_eps=0.0)
    g = v.Context(flags=v.VICP_FLAG_KEEP_GRID, **kw)
    d = v.Context(flags=v.VICP_FLAG_KEEP_GRID | v.VICP_FLAG_NO_GRAPH, **kw)
    s, t = _cloud(3, n)
    other_s, other = _cloud(4, n // 3)
    far = t.clone()   # contents of a later call: points outside the kept grid among them
    far[: n // 10, :3] *= 1.3
    hs, ht = s.cpu().pin_memory(), t.cpu().pin_memory()
    pose0 = torch.eye(4, dtype=torch.float64, device="cuda")
    pose0[0, 3] = 0.05

    def register(c):
        r = c.register_host(hs.numpy(), ht.numpy()) if host else c.register(s, t)
        assert r[0] == 0
        return r

    def look(c):
        nn, d2, nf = c.correspond(s, pose0)
        pose, rmse = pose0.clone(), torch.zeros(1, dtype=torch.float64, device="cuda")
        c.step(s, pose, rmse)
        assert c.sync() == 0
        grid = {k: to_np(x) for k, x in c.get_grid().items()}
        return [to_np(x) for x in (nn, d2, nf, pose, rmse)] + [grid[k] for k in ("keys", "offsets", "root", "ring", "occupancy")] + \
               [np.array([grid["n_target"], grid["n_stored"], grid["dilation_layers"]])]

    def both(call):
        a, b = call(g), call(d)
        for x, y in zip(a, b):
            assert np.array_equal(np.asarray(x), np.asarray(y))

    for _ in range(3):
        both(register)
    assert g.graph_replayed()
    both(look)
    for change in ("build", "dilate", "contents"):
        for c in (g, d):
            if change != "contents":
                c.build_grid(other)
                c.dilate(4 if change == "dilate" else -1)
        if change == "contents":
            (ht if host else t).copy_(far)
        both(register)
        assert g.graph_replayed()
        both(look)
        # and builds after the replay start from clean buffers
        for c in (g, d):
            c.build_grid(other)
            c.dilate()
        both(look)
