"""The size-edge suites of the sieve and of the entry points on the bounds-checked
build, as test_gpu_checked.py does with the parity suites: every store whose
index comes from data, a scan or a counter is checked against its array."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_edge_suites_on_the_checked_build():
    import paper_1810_11966_gb300.build as b
    b.build()
    env = dict(os.environ, JPSI_LIBRARY=b.LIB_CHECKED)
    # (times are those of the ordinary build)
    r = subprocess.run([sys.executable, "-m", "pytest", "tests/test_gpu_sieve.py", "tests/test_gpu_edges.py", "-m", "gpu",
                        "-q", "-x", "-k", "not speed and not pinned", "-p", "no:cacheprovider"],
                       cwd=ROOT, env=env, capture_output=True, text=True, timeout=1800)
    assert r.returncode == 0, r.stdout[-4000:] + r.stderr[-2000:]
    assert " passed" in r.stdout and "failed" not in r.stdout
