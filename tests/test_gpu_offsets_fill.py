"""The offsets array completed for a grid view after a build that writes no entry of the occupancy words without a
point: words whose last voxel is occupied before an empty word, empty scan tiles, and grids that end on a word, inside
one and on a tile of 16384 voxels."""
import numpy as np
import pytest

from gpu_util import assert_grid_equal, gpu_grid, oracle_grid_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [1, 31, 32, 33, 64, 16384, 16385, 16384 * 3, 16384 * 5 + 31])
@pytest.mark.parametrize("which", ["ends_of_words", "last", "first", "few", "many"])
def test_offsets_of_long_rows(nx, which):
    rng = np.random.default_rng(nx)
    v = {"ends_of_words": np.arange(31, nx, 96), "last": np.array([nx - 1] * 3), "first": np.array([0, 0]),
         "few": rng.integers(0, nx, 5), "many": rng.integers(0, nx, min(4 * nx, 30000))}[which]
    if v.size == 0:
        v = np.array([nx - 1])
    t = np.zeros((v.size, 4), np.float32)
    t[:, 0] = v + 0.5
    t[:, 1:3] = 0.5
    ctx, g = gpu_grid(t, L=2, voxel_size=1.0, origin=(0.0, 0.0, 0.0), dims=(nx, 1, 1))
    _, ref = oracle_grid_for(g, t, 2)
    assert_grid_equal(g, ref, t)
    ctx.build_grid(g["_target"])   # and rebuilt over the completed array
    ctx.dilate(2)
    again = ctx.get_grid()
    assert np.array_equal(again["offsets"].view(__import__("torch").int32).cpu().numpy().view(np.uint32), ref["off"])
