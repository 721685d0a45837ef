"""The walks by warps, the runs cut by their drift and the small-city credits under the
bounds-checked build: their tests run in it, and no call reports an index out of range."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
FILES = ["test_gpu_trace_modes.py", "test_gpu_contribution_sparse.py", "test_gpu_contribution_few.py", "test_gpu_iam_sparse.py",
         "test_gpu_batch_delta.py"]


def test_sparse_walks_in_the_checked_build(cuda_lib):
    r = subprocess.run([sys.executable, "-m", "pytest", "-q", "-x", "-p", "no:cacheprovider", "-m", "gpu",
                        *[os.path.join(HERE, f) for f in FILES]], env=dict(os.environ, SA_CHECKED="1"),
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-1000:]
