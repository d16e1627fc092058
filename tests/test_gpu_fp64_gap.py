"""The FP64 solve where the largest eigenvalue is close to the next one, on sums that are exact: rods of eight points
and their matches on a dyadic lattice, rotated against one another by a rational rotation, so that neither the points
nor the sums round and the rotation is known.  Gaps (over |H|) on both sides of what the closed form and its Newton step
can take, det H of both signs.

Tolerance: the residual N q - l q rounds by at most 14 * 2^-53 (four products a row, |N| <= sqrt(3) |H|, and l alike),
N's own entries by 3 * 2^-53; over the gap, doubled from the quaternion to the rotation's entries, 34; what a correction
of at most 1e-9 solved in float leaves is 9 more: 48 * 2^-53 over the gap with the rotation's own rounding."""
from fractions import Fraction as F

import numpy as np
import pytest
import torch

from gpu_util import context, vicp

pytestmark = pytest.mark.gpu

X = [F(k, 2) for k in (-7, -5, -3, -1, 1, 3, 5, 7)]
EVEN = [1, -1, -1, 1, 1, -1, -1, 1]     # orthogonal to X, to ODD and to a constant
ODD = [-1, 1, 1, -1, 1, -1, -1, 1]
TURNS = [(3, 4, 5), (4, -3, 5), (5, 12, 13), (-5, 12, 13), (15, -8, 17), (8, 15, 17)]
FRAMES = [np.array(m, dtype=object) for m in ([[1, -8, 4], [4, 4, 7], [-8, 1, 4]], [[2, -2, 1], [1, 2, 2], [-2, -1, 2]],
                                              [[2, 3, 6], [6, 2, -3], [-3, 6, -2]])]


def _rod(gap, sign, turn, frame, width):
    """Target and source points, both scaled to integers over 2^14, and the rotation of source to target, exactly."""
    r = 1 << 14
    c, s, n = TURNS[turn]
    M = FRAMES[frame]
    d = int(round(float(sum(M[0] * M[0])) ** 0.5))
    assert (M.dot(M.T) == d * d * np.eye(3, dtype=object)).all()
    s1 = float(sum(x * x for x in X))
    if sign > 0:   # H = diag(s1, 8 Y Y, 8 Z Z)
        Y = F(round(r * (gap * s1 / 2 / 8 * (1 + width) / 2) ** 0.5), r)
        Z = F(round(r * (gap * s1 / 2 / 8 - float(Y * Y)) ** 0.5), r)
    else:          # H = diag(s1, 8 Y Y, -8 Z Z)
        Z = F(round(r * width), r)
        Y = F(round(r * (float(Z * Z) + gap * s1 / 2 / 8) ** 0.5), r)
    q = np.array([[n * x, n * Y * e, sign * n * Z * o] for x, e, o in zip(X, EVEN, ODD)], dtype=object)
    p = np.array([[n * x, Y * e, Z * o] for x, e, o in zip(X, EVEN, ODD)], dtype=object)
    A = np.array([[1, 0, 0], [0, c, -s], [0, s, c]], dtype=object)   # (n times a turn about the rod, on y and z)
    p = p.dot(A.T)
    p, q = p.dot(M.T), q.dot(M.T)
    U = np.array([[n, 0, 0], [0, c, s], [0, -s, c]], dtype=object)
    R = M.dot(U).dot(M.T).astype(float) / (n * d * d)
    S = np.array([s1, 8 * float(Y * Y), 8 * sign * float(Z * Z)])
    g = 2 * (S[1] + S[2]) / np.linalg.norm(S)

    def cloud(a):
        out = np.zeros((8, 4), np.float32)
        out[:, :3] = a.astype(float)
        assert all(F(float(out[i, k])) == a[i, k] for i in range(8) for k in range(3))
        return out
    T, P = cloud(q), cloud(p)
    near = np.linalg.norm(P[:, None, :3].astype(float) - T[None, :, :3], axis=2)
    assert (near.argmin(1) == np.arange(8)).all()
    assert max(np.ptp(T[:, :3], axis=0)) < 1024   # one voxel of 1024, and sums of 51 bits about its centre
    return T, P, R, g


CASES = [(t, f, w) for t in range(len(TURNS)) for f in range(len(FRAMES)) for w in (0, 1, 2, 3)]


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("sign", [1, -1])
@pytest.mark.parametrize("gap", [1e-2, 2e-3, 1e-3, 5e-4, 2e-4, 1.2e-4, 5e-5])
def test_rotation_of_rods(gap, sign, batched):
    v = vicp()
    rods = [_rod(gap, sign, t, f, (0.1, 0.3, 0.6, 0.9)[w] if sign > 0 else (0.05, 0.1, 0.15, 0.2)[w])
            for t, f, w in CASES]
    got = []
    if batched:
        b = v.Batch(dilation_layers=1, max_iters=1, flags=v.VICP_BATCH_FLAG_FP64)
        n = np.full(len(rods), 8, np.int32)
        b.build(torch.from_numpy(np.concatenate([r[0] for r in rods])).cuda(), n, np.full(len(rods), 1024, np.float32), None)
        st, T, _, _, each = b.register(torch.from_numpy(np.concatenate([r[1] for r in rods])).cuda(), n)
        assert st == 0 and (each == 0).all()
        got = T
    else:
        for t, p, _, _ in rods:
            ctx = context(voxel_size=2048.0, L=1, origin=(-1024.0,) * 3, dims=(1, 1, 1), flags=v.VICP_FLAG_FP64_SOLVE)
            ctx.build_grid(torch.from_numpy(t).cuda())
            ctx.dilate()
            d = torch.eye(4, dtype=torch.float64, device="cuda")
            ctx.step(torch.from_numpy(p).cuda(), d)
            assert ctx.sync() == 0
            got.append(d.cpu().numpy())
            ctx.close()
    err = [float(np.abs(T[:3, :3] - R).max()) * g / 2.0 ** -53 for T, (_, _, R, g) in zip(got, rods)]
    assert max(err) <= 48, (max(err), int(np.argmax(err)))
