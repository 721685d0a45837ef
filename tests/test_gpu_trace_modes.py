"""The ray-traced accrual's walks: mode 1 is the warp-coherent walk for any receivers, which the
default takes where points are few for the scene's triangles; the work counters are those
of the walk that runs, and no result depends on it."""
import numpy as np
import pytest
import torch

from synth import city as C
from synth.sun import sun_table

pytestmark = pytest.mark.gpu


def _by_mode(B, scene, recv, sun, mode):
    B.sa_set_option(B.SA_OPT_ACCRUAL_TRAVERSAL, mode)
    try:
        return (B.sa_accumulate(scene, recv, sun, 4.0, "accrual_trace"),
                B.sa_work_counters(scene, recv, sun, "accrual_trace"))
    finally:
        B.sa_set_option(B.SA_OPT_ACCRUAL_TRAVERSAL, 0)


def _scene(B, n, extent):
    city = C.city_district(C.SEED_BASE + 91, extent=extent, n_buildings=n)
    m = C.extrude(city)
    return city, B.Scene(m.verts, m.tris, m.tri_building, city.B)


def test_packet_mode_and_its_counters(cuda_lib):
    B = cuda_lib
    _, scene = _scene(B, 100, 600.0)
    st = sun_table(40.7, [172, 200], 9.0, 16.5, 4.0)
    sun = B.Sun(st.dirs, st.day_start)
    grid = B.Receivers.ground_grid(101.0, 83.0, 3.0, 75, 50)
    (a, ca), (b, cb) = (_by_mode(B, scene, grid, sun, mode) for mode in (0, 1))
    assert all(torch.equal(x, y) for x, y in zip(a, b)) and int(a[0].sum()) > 0
    # the grid's groups test a node once for 128 receivers, its warps once a receiver
    assert cb[0] > 8 * ca[0] > 0


# about 29,000 triangles in a plan of 1,500 m; 8 blocks of 8 steps, slopes to 1.7
@pytest.mark.parametrize("n,normals,corner,by_warps", [(700, True, 1.0, True), (20_000, True, 1.0, True),
                                                       (20_000, False, 1.0, True), (80_000, True, 1.0, False),
                                                       (20_000, False, 0.2, False)])
def test_few_points_for_the_triangles_go_by_warps(cuda_lib, n, normals, corner, by_warps):
    B = cuda_lib
    city, scene = _scene(B, 900, 1500.0)
    assert 25_000 < scene.info()["n_tris"] < 33_000
    st = sun_table(40.7, [172], 9.0, 16.5, 8.0)
    sun = B.Sun(st.dirs, st.day_start, 8)
    assert sun.n_blocks == 8 and np.abs(st.dirs[:, :2] / st.dirs[:, 2:]).max() < 2.0
    pos, nrm = C.facade_samples(city, n, 5)
    if not normals:
        pos = np.random.default_rng(4).uniform(0.0, 1500.0 * corner, (n, 3)).astype(np.float32)
        pos[:, 2] *= 0.01
    recv = B.Receivers.points(pos, nrm if normals else None)
    (a, ca), (b, cb) = (_by_mode(B, scene, recv, sun, mode) for mode in (0, 1))
    assert all(torch.equal(x, y) for x, y in zip(a, b)) and int(a[0].sum()) > 0
    assert (ca == cb) == by_warps
    c = B.sa_accumulate(scene, recv, sun, 4.0, "accrual_sam")
    assert all(torch.equal(x, y) for x, y in zip(b, c))


@pytest.mark.parametrize("n", [1, 31, 129, 700])
@pytest.mark.parametrize("doys,step,block_len", [((172,), 4.0, 0), ((355, 20), 3.0, 64), ((80,), 8.0, 1)])
def test_walks_by_warps_equal_the_light_space_map(cuda_lib, n, doys, step, block_len):
    B = cuda_lib
    city, scene = _scene(B, 100, 600.0)
    pos, nrm = C.facade_samples(city, n, 5)
    st = sun_table(40.7, list(doys), 9.0, 16.5, step)
    sun = B.Sun(st.dirs, st.day_start, block_len)
    for normals in (nrm, None):
        recv = B.Receivers.points(pos, normals)
        a, _ = _by_mode(B, scene, recv, sun, 1)
        b = B.sa_accumulate(scene, recv, sun, 4.0, "accrual_sam")
        assert all(torch.equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("doy,t0,t1,step,block_len", [(233, 5.0, 13.0, 5.0, 0), (282, 11.0, 17.0, 15.0, 64),
                                                      (80, 6.0, 18.0, 10.0, 0), (172, 4.6, 19.4, 15.0, 1),
                                                      (355, 8.0, 16.0, 1.0, 33), (172, 8.0, 18.0, 60.0, 7)])
def test_runs_whose_rays_spread_far(cuda_lib, doy, t0, t1, step, block_len):
    """Sunrise, sunset and hours between the steps: runs are cut by their drift, into pieces of
    down to one step, without a change of the results."""
    B = cuda_lib
    city, scene = _scene(B, 100, 600.0)
    st = sun_table(40.7, [doy], t0, t1, step)
    sun = B.Sun(st.dirs, st.day_start, block_len)
    pos, nrm = C.facade_samples(city, 3000, 5)
    for recv in (B.Receivers.points(pos, nrm), B.Receivers.points(pos)):
        a, b = (B.sa_accumulate(scene, recv, sun, step, m) for m in ("accrual_trace", "accrual_sam"))
        assert all(torch.equal(x, y) for x, y in zip(a, b)) and int(a[0].sum()) > 0
    nx, ny, dx = 71, 45, 4.0
    grid = B.Receivers.ground_grid(101.0, 83.0, dx, nx, ny)
    a, c = B.sa_accumulate(scene, grid, sun, step, "accrual_trace"), _by_mode(B, scene, grid, sun, 1)[0]
    xs = np.float32(101.0) + (np.arange(nx, dtype=np.float32) + np.float32(0.5)) * np.float32(dx)
    ys = np.float32(83.0) + (np.arange(ny, dtype=np.float32) + np.float32(0.5)) * np.float32(dx)
    X, Y = np.meshgrid(xs, ys)
    pts = B.Receivers.points(np.stack([X.ravel(), Y.ravel(), np.zeros(nx * ny)], 1).astype(np.float32))
    b = B.sa_accumulate(scene, pts, sun, step, "accrual_sam")
    assert torch.equal(a[0], b[0]) and torch.equal(a[2], b[2])
    assert torch.equal(a[0], c[0]) and torch.equal(a[2], c[2])


@pytest.mark.parametrize("n", [1, 129, 5000])
def test_points_of_a_small_scene(cuda_lib, n):
    """Under 1,000 triangles facade points are taken in their own order."""
    B = cuda_lib
    city = C.city_boxes(C.SEED_BASE + 1)
    m = C.extrude(city)
    assert len(m.tris) < 1000
    scene = B.Scene(m.verts, m.tris, m.tri_building, city.B)
    st = sun_table(40.7, [172, 355], 9.0, 16.0, 7.0)
    sun = B.Sun(st.dirs, st.day_start)
    pos, nrm = C.facade_samples(city, n, 5)
    recv = B.Receivers.points(pos, nrm)
    a, b = (B.sa_accumulate(scene, recv, sun, 7.0, m) for m in ("accrual_trace", "accrual_sam"))
    assert all(torch.equal(x, y) for x, y in zip(a, b)) and (n == 1 or int(a[0].sum()) > 0)
