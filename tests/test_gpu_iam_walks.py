"""The inverse map's source search shares a walk between a block's last step and the next
block's first.  With every block a day of its own no walk is shared, and the masks are the
same bit for bit; groups of cells at their edges, one-step blocks, every number of levels."""
import numpy as np
import pytest
import torch

from synth import city as C
from synth.sun import sun_table

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(1, 1), (16, 8), (17, 9), (63, 41)])
@pytest.mark.parametrize("block_len,levels", [(0, 3), (1, 1), (2, 8), (33, 2)])
def test_shared_walks_equal_separate_ones(cuda_lib, nx, ny, block_len, levels):
    B = cuda_lib
    city = C.city_district(C.SEED_BASE + 23, extent=400.0, n_buildings=60)
    m = C.extrude(city)
    scene = B.Scene(m.verts, m.tris, m.tri_building, city.B)
    st = sun_table(40.7, [172, 355], 9.0, 16.0, 6.0)
    grid = B.Receivers.ground_grid(110.0, 105.0, 2.5, nx, ny)
    j0, K = B.block_partition(st.day_start, block_len)
    own = np.append(j0, j0[-1] + K[-1]).astype(np.int32)        # every block a day
    a = B.Sun(st.dirs, st.day_start, block_len)
    b = B.Sun(st.dirs, own, 64)
    assert a.n_blocks == b.n_blocks == len(j0)
    ma, mb = (B.sa_shadow_masks(scene, grid, s, "iam", iam_levels=levels) for s in (a, b))
    assert torch.equal(ma, mb)
    assert nx < 16 or bool(ma.any())
