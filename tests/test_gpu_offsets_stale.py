"""vicp_offsets_static on a scratch area that holds counts without an occupancy bit, as calls that overlapped or one
that failed half way may leave them: the scan finds that a tile's counts are not this cloud's alone, and the call clears
everything and does its work again.  The scratch is private to its source file, so that file is compiled here once more
together with a function that spoils it, and linked to the library's other objects."""
import ctypes as C
import glob
import os
import subprocess

import numpy as np
import pytest
import torch

import oracle
from gpu_util import to_np, vicp
from paper_2512_04996_gb300 import build, synth

pytestmark = pytest.mark.gpu

SPOIL = """
#include "vicp_static.cu"
extern "C" VICP_API int spoil(long long word, unsigned value, int bit)
{
    unsigned char *base = nullptr;
    if (scratch_address(&base) != VICP_OK)
        return 1;
    if (cudaMemcpy(base + OFF_COUNTS + 4 * word, &value, 4, cudaMemcpyHostToDevice) != cudaSuccess)
        return 2;
    const unsigned occ = 1u << (word & 31);
    return bit && cudaMemcpy(base + OFF_OCC + word / 32 * 4, &occ, 4, cudaMemcpyHostToDevice) != cudaSuccess;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    vicp()   # (built)
    d = tmp_path_factory.mktemp("spoil")
    src, so = os.path.join(d, "spoil.cu"), os.path.join(d, "spoil.so")
    with open(src, "w") as f:
        f.write(SPOIL)
    objs = [o for o in glob.glob(os.path.join(build.BUILD, "*.o")) if os.path.basename(o) != "vicp_static.o"]
    subprocess.check_call([build._nvcc(), *build.NVCC_FLAGS, "-shared", "-cudart", "static", "-o", so, src, *objs])
    return C.CDLL(so)


@pytest.mark.parametrize("bit", [0, 1])
def test_stale_counts(lib, bit):
    p = synth.sphere_plane(seed=9, n=5000)
    grid = oracle.fit_grid(p.target, 0.0, 40)
    ref = oracle.build_grid(grid, p.target, 0)
    t = torch.from_numpy(p.target).cuda()
    o, dims = (C.c_float * 3)(*grid.origin), (C.c_int32 * 3)(*grid.dims)

    def call(n):
        keys = torch.full((n,), -9, dtype=torch.int32, device="cuda")
        off = torch.full((grid.n_voxels + 1,), -9, dtype=torch.int32, device="cuda")
        st = lib.vicp_offsets_static(C.c_void_p(t.data_ptr()), n, o, C.c_float(grid.h), dims, C.c_void_p(keys.data_ptr()),
                                     C.c_void_p(off.data_ptr()),
                                     C.c_void_p(torch.cuda.current_stream().cuda_stream))
        torch.cuda.synchronize()
        assert st == 0
        return to_np(keys), to_np(off)

    voxels = np.unique(ref["keys"][ref["keys"] != ref["keys"][0]])
    for voxel in (int(voxels[0]), int(voxels[len(voxels) // 2]), int(voxels[-1])):
        call(1)   # (its one point's voxel is all that the next call finds to clear)
        assert lib.spoil(C.c_longlong(voxel), C.c_uint(7), bit) == 0
        keys, off = call(5000)
        assert np.array_equal(keys, ref["keys"]) and np.array_equal(off.view(np.uint32), ref["off"])
