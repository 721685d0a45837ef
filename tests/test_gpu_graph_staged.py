"""The direction graph's reduction from staged summaries and from global memory: with bins so
small that every distinct block is an edge of its own, and days that repeat, both equal the
exact accumulation bit for bit.  Numbers of edges and of blocks at the rule's lines and at
the staging's edges, grids at the edges of a CTA's 256 receivers."""
import numpy as np
import pytest
import torch

from synth import city as C
from synth.sun import sun_table

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(1, 1), (255, 1), (256, 1), (257, 1), (50, 31)])
@pytest.mark.parametrize("steps,days,block_len,edges", [(1, 1, 1, 1), (64, 9, 64, 1), (103, 5, 1, 103), (208, 1, 1, 208),
                                                        (209, 1, 1, 209), (230, 6, 1, 230), (421, 7, 1, 421),
                                                        (421, 5, 2, 211)])
def test_reduction_equals_the_exact_accumulation(cuda_lib, nx, ny, steps, days, block_len, edges):
    B = cuda_lib
    city = C.city_district(C.SEED_BASE + 17, extent=400.0, n_buildings=60)
    m = C.extrude(city)
    scene = B.Scene(m.verts, m.tris, m.tri_building, city.B, closed=True)
    day = sun_table(40.7, [172], 9.0, 16.0, 1.0).dirs[:steps]
    assert len(day) == steps
    sun = B.Sun(np.tile(day, (days, 1)), np.arange(days + 1, dtype=np.int32) * steps, block_len)
    grid = B.Receivers.ground_grid(100.0, 120.0, 0.75, nx, ny)
    gross, minutes, cont, n_edges = B.sa_accumulate_graph(scene, grid, sun, 1.0, "accrual_sam", 1e-3)
    assert n_edges == edges
    for a, b in zip((gross, minutes, cont), B.sa_accumulate(scene, grid, sun, 1.0, "accrual_sam")):
        assert torch.equal(a, b)
