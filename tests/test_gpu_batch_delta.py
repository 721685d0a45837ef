"""Batched scenarios put together from the base city's masks against every tile rastered whole
(tile skipping off), bit for bit: variants that only add, only remove, do both or neither,
more changed triangles than one round picks, regions ragged and whole, intervals of
different lengths, one-step blocks, open and closed cities."""
import numpy as np
import pytest
import torch

from synth import city as C
from synth.sun import sun_table

pytestmark = pytest.mark.gpu


def _tower(x, y, side, h):
    return C.extrude(C.City([C.box_footprint(x, y, x + side, y + side)], np.array([h], np.float32))).tri9()


@pytest.mark.parametrize("closed", [True, False])
@pytest.mark.parametrize("block_len", [0, 1])
def test_delta_equals_whole_tiles(cuda_lib, closed, block_len):
    B = cuda_lib
    city = C.city_district(C.SEED_BASE + 55, extent=600.0, n_buildings=100)
    m = C.extrude(city)
    scene = B.Scene(m.verts, m.tris, m.tri_building, city.B, closed=closed)
    grid = B.Receivers.ground_grid(31.0, 17.0, 2.0, 205, 171)
    step = 20.0 if block_len == 1 else 5.0
    suns = []
    for doys in ((172,), (355, 356)):
        st = sun_table(40.7, list(doys), 9.0, 16.0, step)
        suns.append(B.Sun(st.dirs, st.day_start, block_len))
    many = np.concatenate([_tower(140.0 + 9 * (i % 6), 210.0 + 9 * (i // 6), 7.0, 30.0 + 5 * i) for i in range(30)])
    assert many.shape[0] > 256                       # more than one round of towers
    towers = [_tower(200.0, 180.0, 40.0, 250.0), np.zeros((0, 9), np.float32), many, np.zeros((0, 9), np.float32)]
    removed = [[], list(range(10, 60)), [3, 40, 41, 99], []]
    assert int(np.isin(m.tri_building, removed[1]).sum()) > 256
    regions = [(0, 0, 205, 171), (33, 31, 97, 101), (5, 64, 130, 33), (100, 100, 1, 1)]
    out = []
    for skip in (1, 0):
        B.sa_set_option(B.SA_OPT_BATCH_TILE_SKIP, skip)
        try:
            bt = B.Batch(scene, grid, towers, removed, regions, suns)
        finally:
            B.sa_set_option(B.SA_OPT_BATCH_TILE_SKIP, 1)
        counts, impact = bt.run()
        first = counts.clone(), impact.clone()
        bt.run(counts, impact)                       # a second run starts from the base again
        assert torch.equal(first[0], counts) and torch.equal(first[1], impact)
        out.append(first)
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    o = bt.offset(0, 3)
    assert int(out[0][1][:o].abs().sum()) > 0 and int(out[0][1][o:bt.offset(1, 0)].abs().sum()) == 0
