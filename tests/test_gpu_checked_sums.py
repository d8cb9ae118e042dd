"""The files on the sizes at which the kernels change their split (intervals, slices, small
workspaces, blocks of the transfer, MODIT and response kernels), on the bounds-checked build:
after each of the child's tests no index check may have failed."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FILES = ["far_sets", "short_lists", "small_workspace", "slices", "series_edge", "mixed_range", "species_batches",
         "modit_reuse", "modit_short", "response_blocks", "response_sparse", "rt_blocks", "rt_layers"]


@pytest.mark.gpu
def test_splits_on_the_checked_build():
    if os.environ.get("XS_CHECKED") == "1":
        pytest.skip("this process already runs on the checked build")
    p = subprocess.run([sys.executable, "-m", "pytest", "-q", "-x", "-m", "gpu", "-p", "no:cacheprovider"] +
                       [f"tests/test_gpu_{f}.py" for f in FILES], cwd=ROOT, env=dict(os.environ, XS_CHECKED="1"),
                       capture_output=True, text=True, timeout=1500)
    assert p.returncode == 0, p.stdout[-4000:] + p.stderr[-2000:]
    assert " passed" in p.stdout and "failed" not in p.stdout
