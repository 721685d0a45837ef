"""The ray-traced accrual's walks by option: mode 1 is the warp-coherent walk for any receivers,
which is also the default's choice for a thin point set; the work counters are those of the
walk that runs, and no result depends on it."""
import numpy as np
import pytest
import torch

from synth import city as C
from synth.sun import sun_table

pytestmark = pytest.mark.gpu


def test_packet_mode_and_its_counters(cuda_lib):
    B = cuda_lib
    city = C.city_district(C.SEED_BASE + 91, extent=600.0, n_buildings=100)
    m = C.extrude(city)
    scene = B.Scene(m.verts, m.tris, m.tri_building, city.B)
    st = sun_table(40.7, [172, 200], 9.0, 16.5, 4.0)
    sun = B.Sun(st.dirs, st.day_start)
    assert np.abs(st.dirs[:, :2] / st.dirs[:, 2:]).max() < 4.0
    pos, nrm = C.facade_samples(city, 300, 5)
    thin = B.Receivers.points(pos, nrm)                   # a quarter as many points as triangles are more
    assert 4 * 300 < scene.info()["n_tris"]
    grid = B.Receivers.ground_grid(101.0, 83.0, 3.0, 75, 50)
    counts, results = {}, {}
    for name, recv in (("thin", thin), ("grid", grid)):
        for mode in (0, 1):
            B.sa_set_option(B.SA_OPT_ACCRUAL_TRAVERSAL, mode)
            try:
                results[name, mode] = B.sa_accumulate(scene, recv, sun, 4.0, "accrual_trace")
                counts[name, mode] = B.sa_work_counters(scene, recv, sun, "accrual_trace")
            finally:
                B.sa_set_option(B.SA_OPT_ACCRUAL_TRAVERSAL, 0)
        assert all(torch.equal(a, b) for a, b in zip(results[name, 0], results[name, 1])), name
        assert int(results[name, 0][0].sum()) > 0
    assert counts["thin", 0] == counts["thin", 1] != [0, 0, 0, 0]
    # the grid's groups test a node once for 128 receivers, its warps once a receiver
    assert counts["grid", 1][0] > 8 * counts["grid", 0][0] > 0
