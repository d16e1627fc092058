"""The FP64 solve's eigenvector: from the closed form and one FP64 Newton step while the eigenvalue gap allows it, by
Jacobi sweeps below.  Clouds drawn out along a line by 1/eps have a gap of about 2 eps^2 of |H|; the source is the
target moved by less than half the points' spacing, so the matches are known and the update must undo the motion.  A
backward stable solve leaves a rotation error of a few 2^-53 over the gap."""
import numpy as np
import pytest
import torch

from gpu_util import context

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("eps", [1.0, 0.3, 0.1, 3e-2, 1e-2, 6e-3, 3e-3, 1e-3])
def test_drawn_out_clouds(eps, batched):
    from paper_2512_04996_gb300 import vicp as v
    k = np.arange(12)
    x, y, z = np.meshgrid(k, k[:5], k[:4], indexing="ij")
    p = np.stack([x.ravel(), eps * y.ravel(), 1.3 * eps * z.ravel()], 1)
    t = np.zeros((p.shape[0], 4), np.float32)
    t[:, :3] = p
    pose = np.eye(4)
    pose[:3, 3] = [0.01 * eps, -0.02 * eps, 0.03 * eps]
    if batched:
        b = v.Batch(dilation_layers=2, max_iters=1, flags=v.VICP_BATCH_FLAG_FP64)
        c = torch.from_numpy(np.concatenate([t, t])).cuda()
        n = np.array([t.shape[0]] * 2, np.int32)
        b.build(c, n, np.array([0.2 * eps] * 2, np.float32), None)
        st, T, it, rm, each = b.register(c, n, np.stack([pose, pose]))
        assert st == 0 and (each == 0).all() and np.array_equal(T[0], T[1])
        got = T[0]
    else:
        ctx = context(voxel_size=0.2 * eps, L=2, flags=v.VICP_FLAG_FP64_SOLVE)
        c = torch.from_numpy(t).cuda()
        ctx.build_grid(c)
        ctx.dilate()
        d = torch.from_numpy(pose).cuda()
        ctx.step(c, d)
        assert ctx.sync() == 0
        got = d.cpu().numpy()
    H = (p - p.mean(0)).T @ (p - p.mean(0))
    s = np.linalg.svd(H, compute_uv=False)
    gap = 2 * (s[1] + s[2]) / np.linalg.norm(H)
    # (the moved source is rounded to float: 2^-24 of its coordinates, averaged over the points in a rotation
    # whose lever is the cloud's width)
    tol = 40 * 2.0 ** -53 / gap + 12 * 2.0 ** -24 / (eps * np.sqrt(p.shape[0]))
    assert np.abs(got[:3, :3] - np.eye(3)).max() <= tol
