"""A failed search under the differentiable loss, which waits for nothing: the loss and its gradients are NaN, a later
call on the batch raises the failure, and the batch then works as a new one does.  (The failure: the iteration kernel's
grid barrier running out of its time limit, by the library's own test flag.)  And the enqueued search against the
synchronous one."""
import ctypes as C
import gc

import numpy as np
import pytest
import torch

from gpu_util import vicp
from paper_2512_04996_gb300 import synth

pytestmark = pytest.mark.gpu


def _setup(flags=0):
    v = vicp()
    gc.collect()   # (a context that went out of scope frees its memory, and waits for the device, here and not below)
    ps = synth.batched_pairs(seed=77, n_pairs=3, n_min=800, n_max=2500)
    tgt = torch.from_numpy(np.concatenate([p.target for p in ps])).cuda()
    src = torch.from_numpy(np.concatenate([p.source for p in ps])).cuda()
    n_tgt = np.array([p.target.shape[0] for p in ps], np.int32)
    n_src = np.array([p.source.shape[0] for p in ps], np.int32)
    b = v.Batch(dilation_layers=10, flags=flags)
    build = (tgt, n_tgt, None, np.array([p.grid_divisions for p in ps], np.int32))
    b.build(*build)
    T0 = torch.from_numpy(np.ascontiguousarray(np.stack([p.T_gt for p in ps]))).cuda()
    xi = torch.full((3, 6), 0.01, dtype=torch.float64, device="cuda").requires_grad_()
    return v, b, build, src.requires_grad_(), n_src, T0, xi


def _step(v, b, src, n_src, T0, xi, recompute):
    loss = v.point_to_point_loss(xi, src, b, n_src, T0, recompute)
    return (loss, *torch.autograd.grad(loss.sum(), (xi, src)))


@pytest.mark.parametrize("recompute", [False, True])
@pytest.mark.parametrize("after", ["loss", "build", "correspond", "register"])
def test_failed_search_gives_nan_and_is_raised(recompute, after):
    v, b, build, src, n_src, T0, xi = _setup()
    ref = _step(v, b, src, n_src, T0, xi, recompute)
    b.set_flags(v.VICP_BATCH_FLAG_TEST_BARRIER_TIMEOUT)
    loss = v.point_to_point_loss(xi, src, b, n_src, T0, recompute)
    again = v.point_to_point_loss(xi, src, b, n_src, T0, recompute)   # (enqueued before the first has failed)
    gx, gs = torch.autograd.grad(again.sum(), (xi, src), retain_graph=True)
    torch.cuda.synchronize()
    assert torch.isnan(loss).all() and torch.isnan(again).all()
    assert torch.isnan(gx).all() and torch.isnan(gs[:, :3]).all()
    b.set_flags(0)
    if after == "register":
        assert b.register(src.detach(), n_src)[0] == v.VICP_ERR_TIMEOUT
    else:
        with pytest.raises(v.VicpError) as e:
            if after == "loss":
                v.point_to_point_loss(xi, src, b, n_src, T0, recompute)
            elif after == "build":
                b.build(*build)
            else:
                b.correspond(src.detach(), n_src, T0)
        assert e.value.status == v.VICP_ERR_TIMEOUT
    # reported once; then as before, the backward pass of a failed forward among it
    for x, y in zip(_step(v, b, src, n_src, T0, xi, recompute), ref):
        assert torch.equal(x, y)
    for x, y in zip(torch.autograd.grad(again.sum(), (xi, src)), ref[1:]):
        assert torch.equal(x, y)
    assert b.register(src.detach(), n_src)[0] == 0


def test_invalid_matches_are_reported_by_a_later_loss():
    v, b, build, src, n_src, T0, xi = _setup()
    s = src.detach()
    nn, _ = b.correspond(s, n_src, T0)
    ref = b.loss(s, n_src, T0, nn)[0]
    wrong = nn.clone()
    wrong[5] = -1
    b.loss(s, n_src, T0, wrong)
    torch.cuda.synchronize()
    b.loss(s, n_src, T0, nn)   # (its kernel meets the status word)
    torch.cuda.synchronize()
    with pytest.raises(v.VicpError) as e:
        b.loss(s, n_src, T0, nn)
    assert e.value.status == v.VICP_ERR_CUDA
    assert torch.equal(b.loss(s, n_src, T0, nn)[0], ref)


def test_enqueued_search_equals_the_synchronous_one():
    v, b, build, src, n_src, T0, xi = _setup()
    s = src.detach()
    nn, d2 = b.correspond(s, n_src, T0)
    nn2, d22 = torch.full_like(nn, -7), torch.full_like(d2, -7.0)
    n = np.ascontiguousarray(n_src)
    st = v.load_library().vicp_batch_correspond_async(b.handle, s.data_ptr(), n.ctypes.data_as(C.c_void_p),
                                                      T0.data_ptr(), nn2.data_ptr(), d22.data_ptr())
    assert st == 0
    torch.cuda.synchronize()
    assert torch.equal(nn, nn2) and torch.equal(d2, d22)
