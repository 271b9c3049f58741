"""The suites of the readings, of the batch's shares and of both mappings of passes 1 and 2
on the bounds-checked build of the library, in a child process: no index of theirs lies
outside its buffer."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SUITES = ["tests/test_gpu_readings.py", "tests/test_gpu_slow_speeds.py", "tests/test_gpu_batch_shares.py",
          "tests/test_gpu_flat.py", "tests/test_gpu_tiles.py", "tests/test_gpu_graphs_of_eight.py"]


def test_suites_stay_in_bounds_on_the_checked_build():
    from paper_2201_12404_gb300 import build
    lib = build.build_bounds_checked()
    res = subprocess.run([sys.executable, "-m", "pytest", "-x", "-q", "-m", "gpu", "-p", "no:cacheprovider", *SUITES],
                         cwd=ROOT, env=dict(os.environ, LBM_LIBRARY=lib), capture_output=True, text=True, timeout=1800)
    tail = "\n".join((res.stdout + res.stderr).splitlines()[-25:])
    assert res.returncode == 0, tail
    assert "LBM_ERR_BOUNDS" not in res.stdout, tail
