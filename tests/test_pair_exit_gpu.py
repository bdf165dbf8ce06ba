"""CTA pairs of the LM-head: the leader's commits arrive on barriers of both
CTAs, and a CTA may leave only when every arrival at its own shared memory has
landed.  Debug builds check this at the end of each pair (DART_ERR_BOUNDS if
an arrival was not waited for), so the pair cases, with ranges of unequal
length among them, run again under that build."""
import os
import subprocess
import sys

import pytest
import torch

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_arrival_outlives_a_pair():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_13524_gb300 import build
    env = dict(os.environ, DART_TEST_LIBRARY=build.build(debug=True))
    cmd = [sys.executable, "-m", "pytest", "-q", "-x", "-m", "gpu", "-p", "no:cacheprovider",
           "tests/test_debug_gpu.py::test_the_debug_library_is_loaded", "tests/test_lmhead_pair_gpu.py"]
    r = subprocess.run(cmd, cwd=ROOT, env=env, capture_output=True, text=True, timeout=1200)
    assert r.returncode == 0, (r.stdout[-4000:] + r.stderr[-2000:]).strip()
    summary = r.stdout.strip().splitlines()[-1]
    assert " passed" in summary and "skipped" not in summary, summary
