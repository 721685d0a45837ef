"""Makes each device allocation of a call fail in turn (sa_check_fail_alloc, bounds-checked build)
and prints, as one JSON line, how each call ended: a list per call of "same" (the results
of the call without a failure), "oom" or what else.  Used by test_gpu_failing_allocations.py,
which runs it in a process of its own with SA_CHECKED=1."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402
import torch  # noqa: E402

from paper_1907_04435_gb300 import binding as B  # noqa: E402
from synth import city as C  # noqa: E402
from synth import configs  # noqa: E402
from synth.sun import sun_table  # noqa: E402


def same(a, b):
    return len(a) == len(b) and all(torch.equal(x, y) for x, y in zip(a, b))


def every_failure(make, use):
    """make() under the n-th allocation's failure for n = 1, 2, ... until no allocation is left
    to fail; use(made) gives the outputs to compare."""
    want = [t.clone() for t in use(make())]
    ends = []
    for n in range(1, 1000):
        torch.cuda.synchronize()
        B.sa_check_fail_alloc(n)
        try:
            made = make()
            left = B.sa_check_fail_alloc(0)
            end = "same" if same(use(made), want) else "different"
        except B.SAError as err:
            left = B.sa_check_fail_alloc(0)
            end = "oom" if err.status == -3 else str(err)
        if left > 0:
            return ends
        ends.append(end)
    return ends + ["no end"]


def batch():
    w = configs.district_small()
    g = w.ground
    scene = B.Scene(w.mesh.verts, w.mesh.tris, w.mesh.tri_building, w.city.B, closed=True)
    grid = B.Receivers.ground_grid(g.x0, g.y0, g.dx, g.nx, g.ny)
    tower = C.extrude(C.City([C.box_footprint(60.0, 60.0, 90.0, 90.0)], np.array([40.0], np.float32))).tri9()
    suns = [B.Sun(w.sun.dirs, w.sun.day_start)]

    def make():
        return B.Batch(scene, grid, [tower, np.zeros((0, 9), np.float32)], [[], [3, 4]],
                       [(0, 0, g.nx, g.ny), (10, 20, 150, 101)], suns)
    b = make()
    assert 0 < b.n_affected < b.n_items          # tiles that keep the base counts among them
    return every_failure(make, lambda bt: [t.clone() for t in bt.run()])


def ground(method, step, **grid):
    w = configs.district_small()
    g = grid or dict(nx=w.ground.nx, ny=w.ground.ny, dx=w.ground.dx)
    scene = B.Scene(w.mesh.verts, w.mesh.tris, w.mesh.tri_building, w.city.B, closed=True)
    recv = B.Receivers.ground_grid(w.ground.x0, w.ground.y0, g["dx"], g["nx"], g["ny"])
    st = sun_table(40.7, [172], 9.0, 17.0, step)
    sun = B.Sun(st.dirs, st.day_start)
    return every_failure(lambda: B.sa_accumulate(scene, recv, sun, step, method), list)


def points():
    w = configs.district_small()
    scene = B.Scene(w.mesh.verts, w.mesh.tris, w.mesh.tri_building, w.city.B)
    sun = B.Sun(w.sun.dirs, w.sun.day_start)
    recv = B.Receivers.points(w.facade_pos, w.facade_nrm)
    return every_failure(lambda: B.sa_accumulate(scene, recv, sun, 4.0, "accrual_trace"), list)


def gradient():
    pk = configs.park(width=120.0, depth=80.0, dx=1.0, n_buildings=24, band=100.0, step=6.0)
    scene = B.Scene.from_footprints(pk.city.footprints, pk.city.heights, pk.city.band_height)
    grid = B.Receivers.ground_grid(pk.ground.x0, pk.ground.y0, pk.ground.dx, pk.ground.nx, pk.ground.ny)
    sun = B.Sun(pk.sun.dirs, pk.sun.day_start, 8)
    # the sums' order follows the list's: the minutes to 1e-9 of the whole
    return every_failure(lambda: B.sa_height_grad(scene, grid, sun, 6.0), lambda o: [(o[1] / 1e4).round(decimals=6)])


CALLS = {"batch": batch,
         "raster": lambda: ground("accrual_sam", 2.0, nx=800, ny=700, dx=0.6), "raster, one block": lambda: ground("accrual_sam", 30.0),
         "steps by tile": lambda: ground("sweep_raster", 8.0, nx=800, ny=800, dx=0.6),
         "sweep": lambda: ground("sweep_trace", 2.0), "sweep, one block": lambda: ground("sweep_trace", 30.0),
         "traced": lambda: ground("accrual_trace", 2.0), "inverse": lambda: ground("iam", 2.0),
         "points": points, "gradient": gradient}

if __name__ == "__main__":
    print(json.dumps({k: CALLS[k]() for k in (sys.argv[1:] or CALLS)}))
