"""The suites of the streams of lines, the ways a stage is launched, the tiles and the time-step bound on
the bounds-checking build of the library (see test_gpu_bounds_check.py for the others): work items of
several rounds and equal pieces, lines shorter than a chunk, the sum that ends a stage, chained
passes, and both kernels of the time-step bound, without one out-of-range index."""
import os
import re
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("CUDA device required", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_stage_suites_meet_no_out_of_range_index_in_the_bounds_checking_build():
    from paper_2101_05886_gb300 import build
    lib = build.build(check=True)
    env = dict(os.environ, FPGB300_LIBRARY=lib, FPGB300_BOUNDS_AUDIT="1")
    cmd = [sys.executable, "-m", "pytest", "tests/test_gpu_streams.py", "tests/test_gpu_stage_launches.py",
           "tests/test_gpu_set_tile.py", "tests/test_gpu_cfl.py", "tests/test_gpu_cfl_ties.py", "-m", "gpu", "-q",
           "-p", "no:cacheprovider"]
    r = subprocess.run(cmd, cwd=ROOT, env=env, capture_output=True, text=True, timeout=1200)
    tail = (r.stdout + r.stderr)[-4000:]
    assert r.returncode == 0, tail
    passed = re.search(r"(\d+) passed", r.stdout)
    assert passed and int(passed.group(1)) >= 120, tail
