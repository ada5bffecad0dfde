"""The checked build runs the steps through sampled blocks clean (needs a GB300).

On the device it verifies there that every search gives the number of samples at or below its key,
that records and staged samples stay in their areas, and that every hit is at its key's position in
N(v).  The tests named below read the status after every call; they run in a child process with
N2V_CHECKED=1, at the list lengths where these steps change their form.
"""
import os
import subprocess
import sys

import pytest
import torch

pytestmark = pytest.mark.gpu

REPO = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_hub_pairs_and_many_jobs_clean_under_self_checks():
    if not torch.cuda.is_available():
        pytest.skip("CUDA device required")
    r = subprocess.run([sys.executable, "-m", "pytest", "-q", "-x", "-p", "no:cacheprovider", "tests/test_gpu_blocks.py",
                        "tests/test_gpu_instances.py", "tests/test_gpu_serve_many.py", "-k", "not side_by_side"],
                       cwd=REPO, env=dict(os.environ, N2V_CHECKED="1"), stdout=subprocess.PIPE,
                       stderr=subprocess.STDOUT, text=True, timeout=1800)
    assert r.returncode == 0, r.stdout[-5000:]
