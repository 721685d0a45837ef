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


CALLS = {"batch": batch}

if __name__ == "__main__":
    print(json.dumps({k: CALLS[k]() for k in (sys.argv[1:] or CALLS)}))
