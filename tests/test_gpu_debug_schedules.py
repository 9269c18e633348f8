"""Batches, clusters, whole rows and halves, plain and device-counted, under the
debug build: every index check in their kernels and every guard region around
the handle's buffers, both read by each sync of the cases."""

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_schedules_under_the_debug_build():
    from paper_2608_08878_gb300 import build
    build.build_debug()
    files = ["debug_build_checks.py", "test_gpu_batches.py", "test_gpu_clusters.py", "test_gpu_row_schedules.py",
             "test_gpu_graph_rows.py"]
    res = subprocess.run([sys.executable, "-m", "pytest", "-x", "-q", "-m", "gpu"]
                         + [os.path.join(ROOT, "tests", f) for f in files],
                         cwd=ROOT, env=dict(os.environ, DC_LIBRARY="debug"), capture_output=True, text=True, timeout=1500)
    assert res.returncode == 0, res.stdout[-4000:] + res.stderr[-2000:]
    assert " passed" in res.stdout
