"""The bounds-checked build over the suites of the window and dense scan
kernels: as tests/test_gpu_checked.py, in a child process that loads the
checked library, every call must give the oracle's keys and report no index
out of range."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SUITES = ["tests/test_gpu_window.py", "tests/test_gpu_window_segments.py", "tests/test_gpu_dense_scan.py",
          "tests/test_gpu_dense_scan_tail.py", "tests/test_gpu_chunks.py"]


def test_window_and_dense_scan_suites_under_the_checked_build():
    sys.path.insert(0, os.path.join(ROOT, "paper_1704_02272_gb300"))
    import build as pfac_build  # the build script, not the package
    lib = pfac_build.build(checked=True)
    env = dict(os.environ, PFAC_LIB=lib)
    r = subprocess.run([sys.executable, "-m", "pytest", "-q", "-x", "-m", "gpu", "-p", "no:cacheprovider", *SUITES],
                       cwd=ROOT, env=env, capture_output=True, text=True, timeout=3000)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-2000:]
    assert " passed" in r.stdout and "failed" not in r.stdout, r.stdout[-2000:]
