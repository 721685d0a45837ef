"""The inverse map's sources on coarse grids, found by warps: the masks equal those by groups bit
for bit (a low building far off thins out the scene, so that the grid counts as a fine
one).  Patches of cells at their edges, one-step blocks, every number of levels, a low sun."""
import numpy as np
import pytest
import torch

from synth import city as C
from synth.sun import sun_table

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,dx", [(1, 1, 90.0), (8, 4, 50.0), (9, 5, 120.0), (33, 17, 35.0), (3, 40, 40.0)])
@pytest.mark.parametrize("doys,block_len,levels", [((172,), 0, 3), ((355,), 1, 1), ((172, 300), 2, 8), ((80,), 33, 2)])
def test_warps_find_the_sources_of_groups(cuda_lib, nx, ny, dx, doys, block_len, levels):
    B = cuda_lib
    city = C.city_district(C.SEED_BASE + 91, extent=1500.0, n_buildings=900)
    st = sun_table(40.7, list(doys), 9.0, 16.0, 6.0)
    sun = B.Sun(st.dirs, st.day_start, block_len)
    grid = B.Receivers.ground_grid(210.0, 205.0, dx, nx, ny)
    masks = []
    for far in (False, True):
        fps, hs = list(city.footprints), list(city.heights)
        if far:
            fps.append(C.box_footprint(-90000.0, -90000.0, -89990.0, -89990.0))
            hs.append(3.0)
        m = C.extrude(C.City(fps, np.asarray(hs, np.float32), 30.0))
        scene = B.Scene(m.verts, m.tris, m.tri_building, len(fps))
        assert (128.0 * dx * dx * len(m.tris) / np.prod(np.ptp(m.verts[:, :2], axis=0)) > 1600.0) == (not far)
        masks.append(B.sa_shadow_masks(scene, grid, sun, "iam", iam_levels=levels))
    assert torch.equal(masks[0], masks[1])
    assert nx * ny < 16 or bool(masks[0].any())
