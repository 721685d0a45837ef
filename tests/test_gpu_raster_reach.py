"""Triangles that cannot reach the grid are dropped before the ground raster's bins when there
are many (triangle, block) pairs: the masks of a scene equal the OR of the masks of its two
halves, each too small for the rule, with none, few, most or all of it within reach."""
import numpy as np
import pytest
import torch

from synth import city as C
from synth.sun import sun_table

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("closed", [True, False])
@pytest.mark.parametrize("near", [0, 1, 90, 600, 800, 1000])
def test_masks_are_the_or_of_the_halves(cuda_lib, near, closed):
    B = cuda_lib
    rng = np.random.default_rng(near)
    n = 1000
    at = rng.uniform(-40.0, 140.0, (n, 2))
    at[near:] += [3000.0, -2500.0]
    side, h = rng.uniform(1.0, 6.0, n), rng.uniform(2.0, 30.0, n).astype(np.float32)
    order = rng.permutation(n)

    def scene(ids):
        feet = [C.box_footprint(*at[i], *(at[i] + side[i])) for i in ids]
        m = C.extrude(C.City(feet, h[ids]))
        return B.Scene(m.verts, m.tris, m.tri_building, len(ids), closed=closed)

    st = sun_table(40.7, [172], 9.0, 16.0, 1.0)
    sun = B.Sun(st.dirs, st.day_start, 1)                       # one-step blocks
    parts = [scene(order), scene(order[:500]), scene(order[500:])]
    pairs = [s.info()["n_tris"] * len(st.dirs) for s in parts]
    assert pairs[0] >= 4 << 20 > max(pairs[1:])
    grid = B.Receivers.ground_grid(0.0, 0.0, 1.0, 99, 70)
    m = [B.sa_shadow_masks(s, grid, sun, "accrual_sam") for s in parts]
    assert torch.equal(m[0], m[1] | m[2])
    assert not m[0].any() if near == 0 else near == 1 or m[0].any()
    gross, _, _ = B.sa_accumulate(parts[0], grid, sun, 1.0, "accrual_sam")
    bits = sum(((m[0] >> k) & 1).sum(dim=0) for k in range(64))
    assert torch.equal(gross.cpu().flatten().to(torch.int64), bits.cpu().flatten().to(torch.int64))
