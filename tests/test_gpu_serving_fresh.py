"""Serving in a process whose first work is the server's: no lane waits for another's kernels to load."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu


def test_requests_overtake_in_a_fresh_process():
    here = os.path.dirname(os.path.abspath(__file__))
    node = os.path.join(here, "test_gpu_batched_serving.py") + "::test_medium_and_small_requests_overtake_a_large_batch"
    r = subprocess.run([sys.executable, "-m", "pytest", "-q", "-m", "gpu", node], cwd=os.path.dirname(here),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:]
