"""Building contribution over groups of 128 listed cells: regions one cell short of, equal to
and past a group, runs at the edges of 16 and 64 steps, and equal distances (twin buildings)."""
import numpy as np
import pytest

import oracle
from synth import city as C

pytestmark = pytest.mark.gpu


def _dirs(n):
    el = np.radians(np.linspace(20.0, 35.0, n))
    az = np.radians(np.linspace(-6.0, 6.0, n))
    return np.stack([np.cos(el) * np.cos(az), np.cos(el) * np.sin(az), np.sin(el)], 1).astype(np.float32)


@pytest.mark.parametrize("steps", [1, 15, 16, 17, 33, 65])
@pytest.mark.parametrize("cells", [1, 127, 128, 129, 257])
def test_twin_boxes_behind_a_strip_of_cells(cuda_lib, cells, steps):
    """A row of cells deep in the shadow of two coincident boxes at every step: every cell-step
    is cast by both, and its nearest hit, at equal distances, goes to one of them; a third
    box behind, as wide and far higher, is met at every step too and is never the nearest."""
    B = cuda_lib
    width = cells * 0.5
    near = C.box_footprint(10.0, -40.0, 20.0, width + 40.0)
    far = C.box_footprint(25.0, -60.0, 35.0, width + 60.0)
    city = C.City([near, near, far], np.array([30.0, 30.0, 90.0], np.float32))
    mesh = C.extrude(city)
    dirs = _dirs(steps)
    scene = B.Scene(mesh.verts, mesh.tris, mesh.tri_building, 3, closed=True)
    sun = B.Sun(dirs, np.array([0, steps], np.int32))
    grid = B.Receivers.ground_grid(0.0, 0.0, 0.5, 7, cells)
    poly = np.array([[2.0, -1.0], [2.5, -1.0], [2.5, width + 1.0], [2.0, width + 1.0]], np.float32)
    pos = np.stack([np.full(cells, 2.25), (np.arange(cells) + 0.5) * 0.5, np.zeros(cells)], 1).astype(np.float32)
    c_o, _, u_o, u_any = oracle.building_steps(mesh.tri9(), mesh.tri_building, pos, None, dirs,
                                               np.array([0, steps], np.int32), 3)
    # the premise: no ray is near the boundary of any box's shadow
    assert np.all(u_o == 0) and u_any == 0 and np.all(c_o == cells * steps)
    casting, nearest, (over, grazing) = B.sa_building_contribution(scene, grid, sun, poly)
    unit = 0.25 / steps
    assert over == 0 and grazing == 0
    assert np.array_equal(np.round(casting / unit).astype(np.int64), c_o)
    n = np.round(nearest / unit).astype(np.int64)
    assert n[2] == 0 and n[0] + n[1] == cells * steps


@pytest.mark.parametrize("boxes, stride", [(12, 1), (13, 1), (60, 4), (64, 16), (65, 1), (65, 16)])
def test_more_buildings_than_a_cells_list(cuda_lib, boxes, stride):
    """A row of thin boxes, building ids `stride` apart (so that all of them fall into one
    class modulo 4, or modulo 4 and 16): credits pair by pair as the oracle's, and a ray
    that meets more than 64 buildings is refused as before."""
    B = cuda_lib
    x = 8.0 + 4.0 * np.arange(boxes)
    city = C.City([C.box_footprint(a, -60.0, a + 1.5, 80.0) for a in x], (14.0 + 2.0 * x).astype(np.float32))
    mesh = C.extrude(city)
    ids = (np.asarray(mesh.tri_building) * stride).astype(np.int32)
    n = stride * boxes
    dirs, cells = _dirs(5), 40
    scene = B.Scene(mesh.verts, mesh.tris, ids, n, closed=True)
    sun = B.Sun(dirs, np.array([0, 5], np.int32))
    grid = B.Receivers.ground_grid(0.0, 0.0, 0.5, 8, cells)
    poly = np.array([[-1.0, -1.0], [5.0, -1.0], [5.0, 30.0], [-1.0, 30.0]], np.float32)
    if boxes > 64:
        with pytest.raises(B.SAError, match="more than 64 buildings"):
            B.sa_building_contribution(scene, grid, sun, poly)
        return
    gx, gy = np.meshgrid((np.arange(8) + 0.5) * 0.5, (np.arange(cells) + 0.5) * 0.5)
    pos = np.stack([gx.ravel(), gy.ravel(), np.zeros(8 * cells)], 1).astype(np.float32)
    c_o, n_o, u_o, u_any = oracle.building_steps(mesh.tri9(), ids, pos, None, dirs, np.array([0, 5], np.int32), n)
    assert u_o.sum() == 0 and u_any == 0 and c_o.sum() == 8 * cells * 5 * boxes    # the premise
    casting, nearest, (over, grazing) = B.sa_building_contribution(scene, grid, sun, poly)
    unit = 0.25 / 5
    assert over == 0 and grazing == 0
    assert np.array_equal(np.round(casting / unit).astype(np.int64), c_o)
    assert np.array_equal(np.round(nearest / unit).astype(np.int64), n_o)
