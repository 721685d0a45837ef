"""The height gradient's certified flip search against the FP64 search: footprints of up to 8
edges take the first, larger ones the second, so a city whose edges are cut in two or three
by collinear vertices (dyadic coordinates: the same prisms exactly) has the same S and
gradient.  Steps of 4 minutes and of 30 (arcs below and above the series' 0.1 rad), several
days, weights.

Tolerances: a flip's time agrees to about 1e-12 of a step; the two triangulations may decide
a cell on an edge differently, which moves a flip across a step end (continuous in S) --
1e-6 of S and 1e-4 of the gradient's norm leave room for a few such cells among the 3,000."""
import numpy as np
import pytest
import torch

from synth.sun import sun_table

pytestmark = pytest.mark.gpu


def _cut(fp, n):
    """Each edge of the polygon in n equal parts (n = 2 or 4: exact for dyadic corners)."""
    out = []
    for a, b in zip(fp, np.roll(fp, -1, axis=0)):
        out += [a + (b - a) * (k / n) for k in range(n)]
    return np.array(out)


@pytest.mark.parametrize("step,doys", [(4.0, (79,)), (30.0, (172, 20))])
def test_cut_edges_keep_the_gradient(cuda_lib, step, doys):
    B = cuda_lib
    rng = np.random.default_rng(7)
    fps, hs = [], []
    for i in range(5):
        for j in range(4):
            x, y = 40.0 * i - 60.0 + rng.integers(0, 8), 36.0 * j - 40.0 + rng.integers(0, 8)
            w, d = rng.integers(2, 6, 2) * 4.0
            box = np.array([[x, y], [x + w, y + 2.0], [x + w - 2.0, y + d], [x - 2.0, y + d - 2.0]])
            fps.append(box)
            hs.append(float(rng.integers(20, 90)))
    st = sun_table(40.7, list(doys), 9.0, 16.0, step)
    sun = B.Sun(st.dirs, st.day_start)
    grid = B.Receivers.ground_grid(-71.3, -52.7, 3.1, 63, 51)      # ragged 8 x 4 patches
    w = torch.rand(grid.R, generator=torch.Generator().manual_seed(3)).cuda()
    res = []
    for n in (1, 4):
        scene = B.Scene.from_footprints([_cut(f, n) for f in fps], hs)
        g, S = B.sa_height_grad(scene, grid, sun, step, w)
        g2, S2 = B.sa_height_grad(scene, grid, sun, step, w)
        assert float(S) == float(S2) and torch.allclose(g, g2, rtol=1e-6)     # S repeats to the bit
        res.append((float(S), g.double()))
    (S1, g1), (S2, g2) = res
    assert S1 > 0 and float(g1.abs().max()) > 0
    assert abs(S1 - S2) <= 1e-6 * S1
    assert float((g1 - g2).norm()) <= 1e-4 * float(g1.norm())
