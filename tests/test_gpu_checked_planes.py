"""The plane passes under the checked build (see test_gpu_checked.py): the lists of blobs, the first nodes, the
records' nodes and the slots of the partial sums stay in range through steps with blobs on every plane, with
full lists and with more blobs than one window, and every result matches the oracle."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_plane_steps_pass_under_the_index_checks():
    from paper_1212_6427_gb300 import build
    build.build_library()
    build.build_library(checked=True)
    res = subprocess.run([sys.executable, "-m", "pytest", "-q", "-x", "-p", "no:cacheprovider",
                          os.path.join("tests", "test_gpu_plane.py"), os.path.join("tests", "test_gpu_blob_rule.py"),
                          os.path.join("tests", "test_gpu_row_blocks.py"), "-k", "steps or blob or crowded"],
                         cwd=ROOT, env=dict(os.environ, ICM_CHECKED="1"), capture_output=True, text=True, timeout=1200)
    assert res.returncode == 0, res.stdout[-4000:] + res.stderr[-2000:]
    assert " passed" in res.stdout
