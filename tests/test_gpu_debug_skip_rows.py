"""The KPP_DEBUG build on the passes that skip rows, the any-d kernel and the
Lloyd update over ordered points: their index checks (rows, scales and D^2
before the asynchronous copies, positions and points of the order) pass on the
sizes at the edges of warps, blocks and chunks, in a child process that loads
the debug library."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CASES = [
    "tests/test_gpu_skip_rows.py::test_same_as_reading_every_row",
    "tests/test_gpu_skip_rows.py::test_edges_of_the_list",
    "tests/test_gpu_skip_rows.py::test_more_centres_than_have_bounds",
    "tests/test_gpu_skip_rows.py::test_batch_equals_single_seedings",
    "tests/test_gpu_skip_rows.py::test_any_width_same_as_the_streamed_form",
    "tests/test_gpu_hand_over.py::test_given_seeds_and_exact_draws",
    "tests/test_gpu_lloyd_ordered.py",
]


def test_index_checks_hold():
    env = dict(os.environ, KPP_DEBUG="1")
    r = subprocess.run([sys.executable, "-m", "pytest", "-q", "-x", "-m", "gpu", *CASES],
                       capture_output=True, text=True, cwd=ROOT, env=env, timeout=1800)
    assert r.returncode == 0, r.stdout[-4000:] + r.stderr[-2000:]
