"""A captured graph and the workspace it was captured with: calls that grow the workspace between two registrations of
the same clouds (a search or a loss of a larger source cloud, the autotuner) leave the second one equal, bit for bit,
to a context that never replays a graph, and the graph that held the old addresses is not replayed."""
import numpy as np
import pytest
import torch

from gpu_util import vicp
from paper_2512_04996_gb300 import synth

pytestmark = pytest.mark.gpu


def _pairs():
    ps = synth.batched_pairs(seed=71, n_pairs=3, n_min=800, n_max=2500)
    tgt = torch.from_numpy(np.concatenate([p.target for p in ps])).cuda()
    src = torch.from_numpy(np.concatenate([p.source for p in ps])).cuda()
    n_tgt = np.array([p.target.shape[0] for p in ps], np.int32)
    n_src = np.array([p.source.shape[0] for p in ps], np.int32)
    dv = np.array([p.grid_divisions for p in ps], np.int32)
    return tgt, n_tgt, dv, src, n_src


@pytest.mark.parametrize("between", ["correspond", "loss", "tune"])
def test_batch_registration_after_the_workspace_grew(between):
    v = vicp()
    tgt, n_tgt, dv, src, n_src = _pairs()
    b = v.Batch(dilation_layers=10, max_iters=5)
    b.build(tgt, n_tgt, None, dv)
    first = b.register(src, n_src)
    assert first[0] == 0 and b.graph_replayed() == 1
    big, n_big = src.repeat(40, 1), n_src * 40   # (pairs' points mixed: any source will do for a search)
    poses = torch.eye(4, dtype=torch.float64, device="cuda").repeat(3, 1, 1).contiguous()
    shape = -1
    if between == "correspond":
        b.correspond(big, n_big, poses)
    elif between == "loss":
        b.loss(big, n_big, poses, torch.zeros(big.shape[0], dtype=torch.int32, device="cuda"))
        torch.cuda.synchronize()
    else:
        shape, _ = b.tune(big, n_big)
    again = b.register(src, n_src)
    plain = v.Batch(dilation_layers=10, max_iters=5, shape=shape, flags=v.VICP_BATCH_FLAG_NO_GRAPH)
    plain.build(tgt, n_tgt, None, dv)
    ref = plain.register(src, n_src)
    assert again[0] == ref[0] == 0
    assert all(np.array_equal(x, y) for x, y in zip(again[1:], ref[1:]))
    if shape < 0:
        assert all(np.array_equal(x, y) for x, y in zip(again[1:], first[1:]))


@pytest.mark.parametrize("between", ["register_host", "correspond", "build"])
def test_registration_after_the_workspace_grew(between):
    v = vicp()
    small, large = synth.sphere_plane(seed=73, n=30000), synth.sphere_plane(seed=74, n=90000)
    kw = dict(grid_divisions=64, dilation_layers=10, max_iters=5, rmse_eps=0.0)
    ctx = v.Context(flags=v.VICP_FLAG_KEEP_GRID, **kw)
    plain = v.Context(flags=v.VICP_FLAG_KEEP_GRID | v.VICP_FLAG_NO_GRAPH, **kw)
    host = between == "register_host"

    def cloud(a):
        t = torch.from_numpy(a)
        return t.pin_memory() if host else t.cuda()

    s, t, s2, t2 = (cloud(a) for a in (small.source, small.target, large.source, large.target))

    def run(c):
        return c.register_host(s.numpy(), t.numpy()) if host else c.register(s, t)

    first = [run(ctx) for _ in range(3)]
    assert ctx.graph_replayed() == 1
    if host:
        assert ctx.register_host(s2.numpy(), t2.numpy())[0] == 0
    elif between == "correspond":
        ctx.correspond(s2, torch.eye(4, dtype=torch.float64, device="cuda"))
    else:
        ctx.build_grid(t2)
    again = [run(ctx) for _ in range(3)]
    ref = run(plain)
    for r in first + again:
        assert r[0] == ref[0] == 0 and r[2:] == ref[2:] and np.array_equal(r[1], ref[1])
