"""The light-space map stops testing a receiver whose steps are all shadowed, within a chunk of
staged triangles and from one chunk to the next.  Its masks equal those of the fan
traversal, which tests every triangle of a receiver, on an open scene of thin boxes that fill
one light-space tile several chunks deep."""
import numpy as np
import pytest
import torch

from synth import city as C
from synth.sun import sun_table

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 32, 33, 96, 119])
@pytest.mark.parametrize("boxes,doy,step,block_len", [(40, 172, 1.0, 0), (40, 355, 4.0, 64), (90, 80, 2.0, 32),
                                                      (40, 20, 8.0, 1)])
def test_masks_equal_the_fan_traversals(cuda_lib, boxes, n, doy, step, block_len):
    B = cuda_lib
    x = 1.0 + 24.0 * np.arange(boxes) / boxes
    h = 3.0 + 20.0 * ((np.arange(boxes) * 7) % 11) / 10.0
    city = C.City([C.box_footprint(a, 4.0, a + 0.1, 20.0) for a in x], h.astype(np.float32))
    m = C.extrude(city)
    scene = B.Scene(m.verts, m.tris, m.tri_building, boxes)
    assert 4 * n < scene.info()["n_tris"]                       # points by fan
    rng = np.random.default_rng(boxes + n)
    # between the boxes, in front of them and above some of them
    pos = rng.uniform([-4.0, 0.0, 0.0], [30.0, 24.0, 12.0], (n, 3)).astype(np.float32)
    st = sun_table(40.7, [doy], 9.0, 16.5, step)
    sun = B.Sun(st.dirs, st.day_start, block_len)
    recv = B.Receivers.points(pos, None)
    masks = [B.sa_shadow_masks(scene, recv, sun, k) for k in ("accrual_trace", "accrual_sam")]
    assert torch.equal(masks[0], masks[1])
    a, b = (B.sa_accumulate(scene, recv, sun, step, k) for k in ("accrual_trace", "accrual_sam"))
    assert all(torch.equal(p, q) for p, q in zip(a, b))
    if n > 30:
        assert int(a[0].max()) > 0 and int(a[0].min()) < len(st.dirs)
