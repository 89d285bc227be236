"""The checked build of the library (compiled with -DBB_DEBUG: indices taken from the schedule are tested against
their ranges inside the kernels, a failing test records a status instead of touching memory) runs the small parity
cases of the tensor-core kernel without reporting anything.  It stands in for a memory checker."""
import os
import subprocess
import sys

import pytest

from paper_2007_14062_b200 import build as _build

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _run_under_the_checked_build(files, select):
    lib = _build.build(debug=True)
    env = dict(os.environ, BIGBIRD_LIB=lib)
    r = subprocess.run([sys.executable, "-m", "pytest", *(os.path.join(ROOT, "tests", f) for f in files), "-x", "-q", "-m", "gpu",
                        "-k", select, "-p", "no:cacheprovider"],
                       cwd=ROOT, env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-2000:]
    assert " passed" in r.stdout


def test_small_cases_pass_under_the_checked_build():
    _run_under_the_checked_build(["test_parity_gpu.py"], "small_cases and fwd or fully_padded and fwd")


def test_cut_tiles_and_gradients_pass_under_the_checked_build():
    """The tiles that a launch cuts, forward (scratch from the pool and from the fixed array) and backward, and the tensor-core
    gradients at the edges of their schedule, each behind the forward pass."""
    _run_under_the_checked_build(["test_parity_gpu.py", "test_zz_no_alloc.py", "test_bwd_gpu.py"],
                                 "split_tiles or splits_global or in_a_row or leave_no_trace")
