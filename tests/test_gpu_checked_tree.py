"""The sum-tree kernel in the range-checked build: the tests of its forms (every
lane count and leaf, cells past their limits, small classes of batches) run
again in a process with TISSUE_CHECKED=1, where an index out of range is
reported instead of accessed."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_form_runs_clean_in_the_checked_build():
    r = subprocess.run([sys.executable, "-m", "pytest", "-q", "-x", "-p", "no:cacheprovider",
                        "tests/test_gpu_packed_limits.py", "tests/test_gpu_batch_small_classes.py",
                        "tests/test_gpu_sum_tree.py", "-k",
                        "not (test_every_form_matches_oracle and promoter)"],
                       env=dict(os.environ, TISSUE_CHECKED="1"), cwd=ROOT, capture_output=True,
                       text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-4000:] + r.stderr[-2000:]
