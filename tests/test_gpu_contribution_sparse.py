"""Building contribution on coarse grids, whose cells walk by warps: the same credits as by groups
(a low building far off thins out the scene, so that the grid counts as a fine one), and
the oracle's where cells meet more buildings than their lists hold."""
import numpy as np
import pytest

import oracle
from synth import city as C
from synth.sun import sun_table

pytestmark = pytest.mark.gpu


def _contribution(B, footprints, heights, grid, sun, poly):
    m = C.extrude(C.City(footprints, np.asarray(heights, np.float32), 30.0))
    scene = B.Scene(m.verts, m.tris, m.tri_building, len(footprints), closed=True)
    return B.sa_building_contribution(scene, grid, sun, poly)


@pytest.mark.parametrize("nx,ny,dx", [(40, 30, 20.0), (33, 5, 24.0), (9, 7, 150.0), (200, 150, 4.5)])
@pytest.mark.parametrize("doy,t0,t1,step,block_len", [(172, 9.0, 17.0, 4.0, 0), (80, 8.0, 17.0, 12.0, 64),
                                                      (355, 11.0, 13.0, 1.0, 16), (172, 9.0, 17.0, 30.0, 1)])
def test_warps_credit_as_groups_do(cuda_lib, nx, ny, dx, doy, t0, t1, step, block_len):
    B = cuda_lib
    city = C.city_district(C.SEED_BASE + 91, extent=1500.0, n_buildings=900)     # 27,000 triangles
    st = sun_table(40.7, [doy], t0, t1, step)
    sun = B.Sun(st.dirs, st.day_start, block_len)
    grid = B.Receivers.ground_grid(20.0, 30.0, dx, nx, ny)
    e, f = 20.0 + nx * dx, 30.0 + ny * dx
    poly = np.array([[25.0, 20.0], [e, 35.0], [e - 30.0, f], [30.0, f - 20.0]], np.float32)
    far = C.box_footprint(-60000.0, -60000.0, -59990.0, -59990.0)
    hs = list(city.heights)
    a = _contribution(B, city.footprints, hs, grid, sun, poly)
    b = _contribution(B, list(city.footprints) + [far], hs + [3.0], grid, sun, poly)
    assert np.array_equal(a[0], b[0][:-1]) and np.array_equal(a[1], b[1][:-1]) and a[2] == b[2]
    assert b[0][-1] == 0.0 and a[1].sum() > 0.0


@pytest.mark.parametrize("boxes,stride", [(12, 1), (13, 1), (40, 4), (64, 1), (65, 1)])
def test_more_buildings_than_a_cells_list(cuda_lib, boxes, stride):
    B = cuda_lib
    x = 8.0 + 4.0 * np.arange(boxes)
    h = (40.0 + 2.0 * x).astype(np.float32)
    # walls in bands, some 16,000 triangles
    city = C.City([C.box_footprint(a, -100.0, a + 1.5, 140.0) for a in x], h, float(h.sum() / 2000.0))
    mesh = C.extrude(city)
    ids = (np.asarray(mesh.tri_building) * stride).astype(np.int32)
    n, nx, ny, dx = stride * boxes, 8, 10, 6.0
    el, az = np.radians(np.linspace(20.0, 35.0, 17)), np.radians(np.linspace(-6.0, 6.0, 17))
    dirs = np.stack([np.cos(el) * np.cos(az), np.cos(el) * np.sin(az), np.sin(el)], 1).astype(np.float32)
    days = np.array([0, 17], np.int32)
    scene = B.Scene(mesh.verts, mesh.tris, ids, n, closed=True)
    sun = B.Sun(dirs, days)
    grid = B.Receivers.ground_grid(-48.0, 0.0, dx, nx, ny)
    poly = np.array([[-50.0, -10.0], [4.0, -10.0], [4.0, 70.0], [-50.0, 70.0]], np.float32)
    if boxes > 64:
        with pytest.raises(B.SAError, match="more than 64 buildings"):
            B.sa_building_contribution(scene, grid, sun, poly)
        return
    gx, gy = np.meshgrid(-48.0 + (np.arange(nx) + 0.5) * dx, (np.arange(ny) + 0.5) * dx)
    pos = np.stack([gx.ravel(), gy.ravel(), np.zeros(nx * ny)], 1).astype(np.float32)
    c_o, n_o, u_o, u_any = oracle.building_steps(mesh.tri9(), ids, pos, None, dirs, days, n)
    assert u_o.sum() == 0 and u_any == 0 and c_o.sum() == nx * ny * 17 * boxes    # the premise
    casting, nearest, (over, grazing) = B.sa_building_contribution(scene, grid, sun, poly)
    unit = dx * dx / 17
    assert over == 0 and grazing == 0
    assert np.array_equal(np.round(casting / unit).astype(np.int64), c_o)
    assert np.array_equal(np.round(nearest / unit).astype(np.int64), n_o)
