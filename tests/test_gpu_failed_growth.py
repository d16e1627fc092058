"""Calls after one that ran out of memory half way through growing the workspace: wherever the allocator stopped, a call
of the size that worked before works again, with the same bits."""
import numpy as np
import pytest
import torch

from gpu_util import vicp
from paper_2512_04996_gb300 import synth

pytestmark = pytest.mark.gpu


class Pool:
    """An allocator over torch's that can be told to fail after `left` more allocations (None: never)."""

    def __init__(self, v):
        self.live, self.left = {}, None

        @v.ALLOC_FN
        def alloc(nbytes, stream, user):
            if self.left is not None:
                if self.left == 0:
                    return None
                self.left -= 1
            t = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
            self.live[t.data_ptr()] = t
            return t.data_ptr()

        @v.FREE_FN
        def free(ptr, nbytes, stream, user):
            torch.cuda.synchronize()
            self.live.pop(ptr).fill_(0x7F)   # what is read after being given up is not what was there

        self.handle = v.vicp_allocator(alloc, free, None)


def _clouds(n, scale):
    p = synth.sphere_plane(seed=n, n=n)
    s, t = p.source.copy(), p.target.copy()
    s[:, :3] *= scale
    t[:, :3] *= scale
    return torch.from_numpy(s).cuda(), torch.from_numpy(t).cuda()


@pytest.mark.parametrize("flags", ["dense", "sparse", "fp64"])
def test_registration(flags):
    v = vicp()
    fl = {"dense": 0, "sparse": v.VICP_FLAG_SPARSE_GRID, "fp64": v.VICP_FLAG_FP64_SOLVE}[flags]
    small, large = _clouds(3000, 1.0), _clouds(40000, 2.5)

    def context(pool=None):
        return v.Context(v.default_params(voxel_size=0.05, dilation_layers=6, max_iters=3, rmse_eps=0.0, flags=fl),
                         allocator=pool.handle if pool else None)

    ref = context().register(*small)
    assert ref[0] == 0
    for k in range(100):
        pool = Pool(v)
        ctx = context(pool)
        first = ctx.register(*small)
        pool.left = k
        st = ctx.register(*large)[0]
        pool.left = None
        again = ctx.register(*small)
        ctx.close()
        assert pool.live == {}
        for r in (first, again):
            assert r[0] == 0 and r[2:] == ref[2:] and np.array_equal(r[1], ref[1]), k
        if st == 0:
            break
        assert st == v.VICP_ERR_OOM
    assert st == 0 and k > 10


def test_a_failed_build_leaves_no_grid():
    v = vicp()
    small, large = _clouds(3000, 1.0), _clouds(40000, 2.5)
    pool = Pool(v)
    ctx = v.Context(v.default_params(voxel_size=0.05, dilation_layers=6), allocator=pool.handle)
    ctx.build_grid(small[1])
    ctx.dilate()
    pool.left = 3
    with pytest.raises(v.VicpError) as e:
        ctx.build_grid(large[1])
    assert e.value.status == v.VICP_ERR_OOM
    pose = torch.eye(4, dtype=torch.float64, device="cuda")
    for call in (lambda: ctx.step(small[0], pose), lambda: ctx.correspond(small[0], pose), lambda: ctx.dilate()):
        with pytest.raises(v.VicpError) as e:
            call()
        assert e.value.status == v.VICP_ERR_STATE
    ctx.close()


@pytest.mark.parametrize("what", ["search", "build"])
def test_batch(what):
    v = vicp()
    def case(seed, lo, hi):
        ps = synth.batched_pairs(seed=seed, n_pairs=3, n_min=lo, n_max=hi)
        return [torch.from_numpy(np.concatenate([getattr(p, a) for p in ps])).cuda() for a in ("source", "target")] + \
               [np.array([getattr(p, a).shape[0] for p in ps], np.int32) for a in ("source", "target")]
    s, t, ns, nt = case(81, 800, 2500)
    S, T, NS, NT = case(82, 9000, 20000)
    small_div, large_div = np.full(3, 32, np.int32), np.full(3, 64, np.int32)
    ref = None
    for k in range(100):
        pool = Pool(v)
        b = v.Batch(v.batch_default_params(max_iters=3, dilation_layers=6), allocator=pool.handle)
        b.build(t, nt, None, small_div)
        first = b.register(s, ns)
        pool.left = k
        st = 0
        try:
            if what == "search":
                b.correspond(s.repeat(30, 1), ns * 30, torch.eye(4, dtype=torch.float64, device="cuda").repeat(3, 1, 1))
            else:
                b.build(T, NT, None, large_div)
                st = b.register(S, NS)[0]
        except v.VicpError as e:
            st = e.status
        pool.left = None
        if what == "build":
            b.build(t, nt, None, small_div)
        again = b.register(s, ns)
        b.close()
        assert pool.live == {}
        ref = ref or first
        for r in (first, again):
            assert r[0] == 0 and all(np.array_equal(x, y) for x, y in zip(r[1:], ref[1:])), k
        if st == 0:
            break
        assert st == v.VICP_ERR_OOM
    assert st == 0 and k > 4


@pytest.mark.parametrize("batched", [False, True])
def test_a_host_registration_that_gave_its_target_copy_up(batched):
    v = vicp()
    (s, t), (S, T) = _clouds(3000, 1.0), _clouds(40000, 1.0)
    pool = Pool(v)
    pose = torch.eye(4, dtype=torch.float64, device="cuda")
    if batched:
        b = v.Batch(v.batch_default_params(max_iters=2), allocator=pool.handle)
        run = lambda x, y: b.register_host(x.cpu().numpy(), [x.shape[0]], y.cpu().numpy(), [y.shape[0]], None, [32])[0]
        look = lambda: b.correspond(s, [s.shape[0]], pose[None].contiguous())
    else:
        b = v.Context(v.default_params(grid_divisions=32, max_iters=2), allocator=pool.handle)
        run = lambda x, y: b.register_host(x.cpu().numpy(), y.cpu().numpy())[0]
        look = lambda: b.step(s, pose.clone())
    assert run(s, t) == 0
    look()
    pool.left = 1   # the source's copy fits, the target's does not
    assert run(S, T) == v.VICP_ERR_OOM
    pool.left = None
    with pytest.raises(v.VicpError) as e:
        look()
    assert e.value.status == v.VICP_ERR_STATE
    assert run(s, t) == 0
    look()
    b.close()
    assert pool.live == {}
