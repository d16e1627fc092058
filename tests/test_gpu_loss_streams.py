"""The differentiable loss on another stream than the batch's: what the caller's stream has yet to compute is waited
for, and what the batch's stream computes is there for the caller's."""
import numpy as np
import pytest
import torch

from gpu_util import vicp
from paper_2512_04996_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("recompute", [False, True])
def test_inputs_and_results_across_streams(recompute):
    v = vicp()
    ps = synth.batched_pairs(seed=79, n_pairs=3, n_min=800, n_max=2500)
    tgt = torch.from_numpy(np.concatenate([p.target for p in ps])).cuda()
    src = torch.from_numpy(np.concatenate([p.source for p in ps])).cuda()
    n = np.array([p.source.shape[0] for p in ps], np.int32)
    T0 = torch.from_numpy(np.ascontiguousarray(np.stack([p.T_gt for p in ps]))).cuda()
    xi0 = torch.linspace(-0.02, 0.03, 18, dtype=torch.float64, device="cuda").reshape(3, 6)
    b = v.Batch(dilation_layers=10)
    b.build(tgt, np.array([p.target.shape[0] for p in ps], np.int32), None,
            np.array([p.grid_divisions for p in ps], np.int32))

    def step(delay):
        if delay:   # (some milliseconds before xi and the source points are there)
            torch.cuda._sleep(20_000_000)
        xi = (xi0 * 1.0).requires_grad_()
        s = (src * 1.0).requires_grad_()
        loss = v.point_to_point_loss(xi, s, b, n, T0, recompute)
        gx, gs = torch.autograd.grad(loss.sum(), (xi, s))
        return loss.detach() * 1.0, gx * 1.0, gs * 1.0

    ref = step(False)
    torch.cuda.synchronize()
    other = torch.cuda.Stream()
    for _ in range(3):
        with torch.cuda.stream(other):
            out = step(True)
        other.synchronize()
        for x, y in zip(out, ref):
            assert torch.equal(x, y)
