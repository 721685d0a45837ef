"""The ray-traced methods cut into items.  The accrual's grouped traversal and its fan traversal
(thin point sets) take the light-space map's FP32 decisions on every triangle, so on an open
scene their masks equal the map's bit for bit; the sweep's pieces do not change its bits.
Sizes at the edges of groups (128 points, 16 x 8 cells), one-step and 64-step blocks, several
days, a low sun, scenes of 0, 1 and 2 triangles."""
import numpy as np
import pytest
import torch

from synth import city as C
from synth.sun import sun_table

pytestmark = pytest.mark.gpu


def _city(n):
    return C.city_district(C.SEED_BASE + 91, extent=600.0, n_buildings=n)


def _scene(B, city):
    m = C.extrude(city)
    return B.Scene(m.verts, m.tris, m.tri_building, city.B)


def _same(B, scene, recv, sun, step, methods):
    out = [B.sa_accumulate(scene, recv, sun, step, m) for m in methods]
    assert all(torch.equal(a, b) for o in out[1:] for a, b in zip(out[0], o))
    masks = [B.sa_shadow_masks(scene, recv, sun, m) for m in methods]
    assert all(torch.equal(masks[0], m) for m in masks[1:])
    # progressive accumulation doubles the gross counts and keeps the longest run
    g, mi, c = (t.clone() for t in out[0])
    B.sa_accumulate(scene, recv, sun, step, methods[0], accumulate_into=True, gross=g, minutes=mi, continuous=c)
    assert torch.equal(g, 2 * out[0][0]) and torch.equal(c, out[0][2])
    return out[0]


@pytest.mark.parametrize("n", [1, 31, 128, 129, 700, 5000])
@pytest.mark.parametrize("doys,step,block_len", [((172,), 4.0, 0), ((355, 20), 3.0, 64), ((80,), 8.0, 1)])
def test_point_groups_equal_the_light_space_map(cuda_lib, n, doys, step, block_len):
    B = cuda_lib
    city = _city(100)
    scene = _scene(B, city)                    # about 3,000 triangles: 700 points and fewer by fan
    assert 4 * 700 < scene.info()["n_tris"] < 4 * 5000
    pos, nrm = C.facade_samples(city, n, 5)
    st = sun_table(40.7, list(doys), 9.0, 16.5, step)
    sun = B.Sun(st.dirs, st.day_start, block_len)
    for normals in (nrm, None):
        g, _, _ = _same(B, scene, B.Receivers.points(pos, normals), sun, step, ("accrual_trace", "accrual_sam"))
    assert n < 100 or int(g.sum()) > 0


@pytest.mark.parametrize("nx,ny", [(1, 1), (16, 8), (17, 9), (75, 50)])
def test_grid_groups_equal_the_same_points(cuda_lib, nx, ny):
    B = cuda_lib
    scene = _scene(B, _city(100))
    st = sun_table(40.7, [172, 300], 9.0, 16.5, 4.0)
    sun = B.Sun(st.dirs, st.day_start)
    grid = B.Receivers.ground_grid(101.0, 83.0, 3.0, nx, ny)
    a = _same(B, scene, grid, sun, 4.0, ("accrual_trace",))
    xs = np.float32(101.0) + (np.arange(nx, dtype=np.float32) + np.float32(0.5)) * np.float32(3.0)
    ys = np.float32(83.0) + (np.arange(ny, dtype=np.float32) + np.float32(0.5)) * np.float32(3.0)
    X, Y = np.meshgrid(xs, ys)
    pts = B.Receivers.points(np.stack([X.ravel(), Y.ravel(), np.zeros(nx * ny, np.float32)], 1))
    b = B.sa_accumulate(scene, pts, sun, 4.0, "accrual_sam")
    assert all(torch.equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("n_tris", [0, 1, 2])
def test_tiny_scenes(cuda_lib, n_tris):
    B = cuda_lib
    v = np.array([[0, 0, 10], [20, 0, 10], [20, 20, 10], [0, 20, 10]], np.float32)
    scene = B.Scene(v, np.array([[0, 1, 2], [0, 2, 3]], np.int32)[:n_tris], np.zeros(n_tris, np.int32), 1)
    st = sun_table(40.7, [172], 11.0, 13.0, 2.0)
    sun = B.Sun(st.dirs, st.day_start)
    p = np.random.default_rng(1).uniform(-10, 30, (400, 3)).astype(np.float32)
    g, _, _ = _same(B, scene, B.Receivers.points(p), sun, 2.0, ("accrual_trace", "accrual_sam"))
    assert (int(g.sum()) > 0) == (n_tris > 0)


@pytest.mark.parametrize("nx,ny", [(5, 3), (64, 40)])
def test_sweep_pieces_keep_the_bits(cuda_lib, nx, ny):
    B = cuda_lib
    scene = _scene(B, _city(60))
    st = sun_table(40.7, [172, 300], 9.0, 16.5, 3.0)
    grid = B.Receivers.ground_grid(101.0, 83.0, 3.0, nx, ny)
    # blocks of 60, 64, 7 and 1 steps are cut into 16, 16, 7 and 1 pieces
    out = [_same(B, scene, grid, B.Sun(st.dirs, st.day_start, k), 3.0, ("sweep_trace",)) for k in (60, 64, 7, 1)]
    assert all(torch.equal(a, b) for o in out[1:] for a, b in zip(out[0], o))
