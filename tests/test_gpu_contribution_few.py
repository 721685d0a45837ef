"""Building contribution's credits on both sides of the line at 256 buildings, under which a warp
adds them up first: the same city with its ids as they are and spread over 257."""
import numpy as np
import pytest

from synth import city as C
from synth.sun import sun_table

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,block_len", [(64, 64, 0), (33, 5, 64), (1, 1, 7)])
def test_credits_by_warp_equal_credits_by_cell(cuda_lib, nx, ny, block_len):
    B = cuda_lib
    city = C.city_boxes(C.SEED_BASE + 1)
    m = C.extrude(city)
    st = sun_table(40.7, [172, 355], 9.0, 16.0, 3.0)
    sun = B.Sun(st.dirs, st.day_start, block_len)
    grid = B.Receivers.ground_grid(40.0, 35.0, 2.0, nx, ny)
    e, f = 40.0 + 2.0 * nx, 35.0 + 2.0 * ny
    poly = np.array([[40.0, 35.0], [e, 35.0], [e, f], [40.0, f]], np.float32)
    few = B.sa_building_contribution(B.Scene(m.verts, m.tris, m.tri_building, city.B), grid, sun, poly)
    ids = (np.asarray(m.tri_building) * 17 + 1).astype(np.int32)
    many = B.sa_building_contribution(B.Scene(m.verts, m.tris, ids, 257), grid, sun, poly)
    at = np.arange(city.B) * 17 + 1
    assert np.array_equal(few[0], many[0][at]) and np.array_equal(few[1], many[1][at]) and few[2] == many[2]
    assert np.delete(many[0], at).sum() == 0.0 and (nx == 1 or few[1].sum() > 0.0)
