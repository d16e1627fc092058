"""The number of global searches, written by the search kernel, in a counter of any alignment (a four-byte field of a
packed record, say), for both stores and for clouds with and without near queries searched by rows."""
import ctypes as C

import numpy as np
import pytest
import torch

from gpu_util import context, vicp
from paper_2512_04996_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [0, 1, 2, 3])
@pytest.mark.parametrize("divisions", [32, 64])
def test_counter_of_any_alignment(divisions, offset):
    v = vicp()
    lib = v.load_library()
    p = synth.sphere_plane(seed=5, n=20000)
    s, t = torch.from_numpy(p.source).cuda(), torch.from_numpy(p.target).cuda()
    pose = torch.eye(4, dtype=torch.float64, device="cuda")
    ctx = context(divisions=divisions)
    ctx.build_grid(t)
    ctx.dilate()
    ctx.fixed_build(t, ctx.memory_report()["max_voxel_count"])
    nn, d2, nf = ctx.correspond(s, pose)
    want = int(nf[0])
    assert want > 0
    for call in (lib.vicp_correspond, lib.vicp_fixed_correspond):
        record = torch.full((16,), 0xAB, dtype=torch.uint8, device="cuda")
        n2, e2 = torch.empty_like(nn), torch.empty_like(d2)
        assert call(ctx.handle, s.data_ptr(), s.shape[0], pose.data_ptr(), n2.data_ptr(), e2.data_ptr(),
                    C.c_void_p(record.data_ptr() + 4 + offset)) == 0
        assert ctx.sync() == 0
        r = record.cpu().numpy()
        assert int(r[4 + offset:8 + offset].copy().view(np.int32)[0]) == want
        assert (np.delete(r, range(4 + offset, 8 + offset)) == 0xAB).all()
        assert torch.equal(n2, nn) and torch.equal(e2, d2)
