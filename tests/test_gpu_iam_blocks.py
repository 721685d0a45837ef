"""The inverse map draws all blocks in one launch: several days at once equal the days one by
one accumulated into the same buffers, and its masks hold the counted steps (blocks of 60, 7
and 1 steps, ragged 8 x 4 patches, cells smaller and larger than a step's shadow motion)."""
import numpy as np
import pytest
import torch

from parity import block_sizes, unpack_masks, workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("block_len", [0, 7, 1])
@pytest.mark.parametrize("dx", [0.25, 5.0])
def test_all_blocks_at_once(cuda_lib, block_len, dx):
    B = cuda_lib
    w = workload("district_small", doys=(172, 300, 20), step=12.0, n_facade=0)
    scene = B.Scene(w.mesh.verts, w.mesh.tris, w.mesh.tri_building, w.city.B)
    grid = B.Receivers.ground_grid(200.0, 180.0, dx, 53, 39)
    sun = B.Sun(w.sun.dirs, w.sun.day_start, block_len)
    got = B.sa_accumulate(scene, grid, sun, 12.0, "iam")
    acc = [torch.zeros(grid.R, dtype=t.dtype, device="cuda") for t in got]
    ds = w.sun.day_start
    for a, b in zip(ds[:-1], ds[1:]):
        day = B.Sun(w.sun.dirs[a:b], np.array([0, b - a], np.int32), block_len)
        B.sa_accumulate(scene, grid, day, 12.0, "iam", accumulate_into=True, gross=acc[0], minutes=acc[1],
                        continuous=acc[2])
    assert all(torch.equal(x, y) for x, y in zip(got, acc)) and int(got[0].sum()) > 0
    bits = unpack_masks(B.sa_shadow_masks(scene, grid, sun, "iam"), block_sizes(ds, block_len))
    assert np.array_equal(bits.sum(1, dtype=np.int64), got[0].cpu().numpy())
