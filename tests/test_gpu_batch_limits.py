"""A batch with more items than 32 bits count: one tile and 65,536 one-step blocks, which the
tower of each of 65,537 variants shadows at every step.  It is made without base masks, by
whole tiles (sa_batch_create's limit of 64M items)."""
import numpy as np
import pytest
import torch

from synth import city as C
from synth.sun import sun_table

pytestmark = pytest.mark.gpu


def test_items_past_32_bits(cuda_lib):
    B = cuda_lib
    V, S = 65537, 65536                            # V x S is 2^32 + 2^16
    st = sun_table(40.7, list(range(1, 151)), 9.0, 16.5, 1.0)
    assert st.S >= S
    days = np.searchsorted(st.day_start, S, side="right") - 1
    start = np.append(st.day_start[:days + 1], S).astype(np.int32) if st.day_start[days] < S else st.day_start[:days + 1]
    sun = B.Sun(st.dirs[:S], start, 1)
    assert sun.n_blocks == S
    v = np.array([[0, 0, 5], [1, 0, 5], [0, 1, 5]], np.float32)
    scene = B.Scene(v, np.array([[0, 1, 2]], np.int32), np.zeros(1, np.int32), 1)
    grid = B.Receivers.ground_grid(0.0, 0.0, 1.0, 32, 32)
    tower = C.extrude(C.City([C.box_footprint(10.0, 10.0, 14.0, 14.0)], np.array([30.0], np.float32))).tri9()
    batch = B.Batch(scene, grid, [tower] * V, [np.zeros(0, np.int32)] * V, [(0, 0, 32, 32)] * V, [sun])
    assert batch.n_items == batch.n_affected == V and batch.n_out == V * 32 * 32
    torch.cuda.synchronize()
    del batch
    # the same with one variant still goes by the masks
    one = B.Batch(scene, grid, [tower], [np.zeros(0, np.int32)], [(0, 0, 32, 32)], [sun])
    counts, impact = one.run()
    g, _, _ = B.sa_accumulate(scene, grid, sun, 1.0, "accrual_sam")
    assert torch.equal(counts - impact, g) and int(impact.max()) > 0
