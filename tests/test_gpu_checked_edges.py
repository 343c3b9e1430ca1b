"""The checked build (see test_gpu_checked.py) over the tests of the kernels' edges: the column
series, the warp-per-pair adjoint (whose plain adds rely on rows inside the window), split
images, coarse spans and fast receivers."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
EDGES = ["test_gpu_series.py", "test_gpu_series16.py", "test_gpu_adjoint2d.py", "test_gpu_splits.py",
         "test_gpu_split_cost.py", "test_gpu_spans.py", "test_gpu_motion_terms.py"]


def test_checked_build_edge_cases_leave_status_clear():
    from paper_2101_05888_gb300 import build
    build.build(checked=True)
    r = subprocess.run([sys.executable, "-m", "pytest", "-x", "-q", "-m", "gpu", "-p", "no:cacheprovider",
                        "-k", "not solve and not cost_the_host",
                        *[os.path.join("tests", f) for f in EDGES]],
                       cwd=ROOT, env=dict(os.environ, SAS_CHECKED="1"), capture_output=True, text=True, timeout=1800)
    print(r.stdout[-3000:])
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
