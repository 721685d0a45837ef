"""What the calls do when device memory runs out: in the bounds-checked build each of their
allocations is made to fail in turn.  Runs in a process of its own."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def _run(*names):
    r = subprocess.run([sys.executable, os.path.join(HERE, "failing_allocations.py"), *names],
                       env=dict(os.environ, SA_CHECKED="1"), capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    return json.loads(r.stdout.strip().splitlines()[-1])


def test_a_batch_does_without_the_base_masks(cuda_lib):
    """Whatever allocation of sa_batch_create fails once the masks are taken, or fails to take
    them, the batch is made without them, and its tiles that no change reaches keep the
    base counts."""
    ends = _run("batch")["batch"]
    first = ends.index("same")
    assert set(ends[:first]) <= {"oom"} and first <= 4         # towers, removed buildings, counter, masks
    assert len(ends) > 12 and set(ends[first:]) == {"same"}


def test_calls_go_on_with_less_memory(cuda_lib):
    """The summaries, masks, sources and bins of many blocks are taken for fewer at a time when they
    do not fit, down to paths that need none; any other failure is reported, and no
    result is wrong."""
    fewer = {"raster": 2, "raster, one block": 1, "steps by tile": 1, "sweep": 1, "sweep, one block": 1, "traced": 1,
             "inverse": 2, "points": 3, "gradient": 1}      # allocations that a call does without
    ends = _run(*fewer)
    for name, n in fewer.items():
        assert set(ends[name]) <= {"same", "oom"} and ends[name].count("same") >= n, (name, ends[name])
