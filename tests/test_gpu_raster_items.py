"""The ground raster by items (a CTA per tile, block and piece of a block) against the raster
by tiles (the fixed-scratch entry point), bit for bit: grids on both sides of every rule
that cuts the work (pieces per block, bins filled directly or counted first, blocks per
chunk), ragged tiles, one-step blocks, several days, open and closed scenes.  Both take the
same FP32 decisions, so counts are equal without a tolerance."""
import numpy as np
import pytest
import torch

from parity import assert_bits_parity, block_sizes, cached_oracle, unpack_masks, workload
from synth import city as C
from synth.sun import sun_table

pytestmark = pytest.mark.gpu


def _scene(B, n, closed):
    city = C.city_district(C.SEED_BASE + 77, extent=700.0, n_buildings=n) if n > 1 else C.City(
        [C.box_footprint(20.0, 20.0, 45.0, 40.0)], np.array([35.0], np.float32))
    m = C.extrude(city)
    return B.Scene(m.verts, m.tris, m.tri_building, city.B, closed=closed)


@pytest.mark.parametrize("n,nx,ny,doys,step,block_len,closed", [
    (1, 1, 1, (172,), 1.0, 0, True),              # one cell; bins filled directly
    (1, 33, 31, (172,), 2.0, 64, False),          # blocks of 61; four pieces
    (200, 65, 64, (172,), 4.0, 1, False),         # one-step blocks: empty pieces
    (200, 97, 33, (172, 173, 355), 4.0, 7, True),
    (200, 640, 320, (172,), 1.0, 0, True),        # 200 tiles x 8 blocks: 1,600 items, two pieces
    (200, 768, 320, (172,), 1.0, 0, False),       # 240 tiles x 8 blocks: 1,920 items, one piece
    (210, 40, 70, tuple(range(100, 190)), 4.0, 30, True),   # 360 blocks in one chunk
])
def test_items_equal_tiles(cuda_lib, n, nx, ny, doys, step, block_len, closed):
    B = cuda_lib
    scene = _scene(B, n, closed)
    st = sun_table(40.7, list(doys), 9.0, 16.0, step)
    sun = B.Sun(st.dirs, st.day_start, block_len)
    grid = B.Receivers.ground_grid(11.0, 7.5, 1.0, nx, ny)
    out = [torch.zeros(grid.R, dtype=d, device="cuda") for d in (torch.int32, torch.float32, torch.int32)]
    B.sa_accumulate_grid_noalloc(scene, grid, sun, step, *out)
    got = B.sa_accumulate(scene, grid, sun, step, "accrual_sam")
    assert all(torch.equal(a, b) for a, b in zip(out, got))
    # progressive accumulation on top of both
    B.sa_accumulate_grid_noalloc(scene, grid, sun, step, *out, accumulate_into=True)
    B.sa_accumulate(scene, grid, sun, step, "accrual_sam", accumulate_into=True, gross=got[0], minutes=got[1],
                    continuous=got[2])
    assert all(torch.equal(a, b) for a, b in zip(out, got))
    # the masks hold the same steps
    bits = unpack_masks(B.sa_shadow_masks(scene, grid, sun, "accrual_sam"), block_sizes(st.day_start, block_len))
    assert np.array_equal(2 * bits.sum(1, dtype=np.int64), got[0].cpu().numpy())


@pytest.mark.parametrize("nx,ny", [(90, 70), (32 * 38, 32 * 16)])    # by item; 608 tiles: by tile
def test_per_step_raster_equals_the_accrual_raster(cuda_lib, nx, ny):
    B = cuda_lib
    scene = _scene(B, 200, True)
    st = sun_table(40.7, [172, 300], 9.0, 16.0, 4.0)
    sun = B.Sun(st.dirs, st.day_start)
    grid = B.Receivers.ground_grid(-200.0, 7.5, 1.0, nx, ny)
    a = B.sa_accumulate(scene, grid, sun, 4.0, "accrual_sam")
    b = B.sa_accumulate(scene, grid, sun, 4.0, "sweep_raster")
    assert all(torch.equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("closed", [True, False])
def test_low_sun_tiles_that_fill_up(cuda_lib, closed):
    """A December afternoon: a tile's bins hold many batches of triangles and its rows fill up
    before the last, which then are skipped; step masks against the oracle."""
    B = cuda_lib
    w = workload("district_small", n_buildings=160, nx=100, ny=90, n_facade=0, doys=(355,), t0=14.0, t1=16.6, step=3.0)
    scene = B.Scene(w.mesh.verts, w.mesh.tris, w.mesh.tri_building, w.city.B, closed=closed)
    sun = B.Sun(w.sun.dirs, w.sun.day_start, 64)
    g = w.ground
    grid = B.Receivers.ground_grid(g.x0, g.y0, g.dx, g.nx, g.ny)
    bits, near = cached_oracle("low_sun", w, "ground")
    tiles = bits.reshape(g.ny, g.nx, -1)
    assert tiles[32:64, 96:].all(axis=(0, 1)).sum() > 40      # a tile wholly shadowed at most steps
    got = unpack_masks(B.sa_shadow_masks(scene, grid, sun, "accrual_sam"), block_sizes(w.sun.day_start, 64))
    assert_bits_parity(got, bits, near)
