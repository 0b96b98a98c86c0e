"""The host code that plans and launches chi, linked against a CUDA runtime that
records what it is asked for (_host_launches.cpp): no GPU."""
import glob
import os
import subprocess

import pytest

from paper_1806_10889_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    B.build()
    objs = [o for o in glob.glob(os.path.join(B.OUT, "*.o")) if not o.endswith("_checked.o")]
    if not objs:  # a library without its objects
        B.build(force=True)
        objs = [o for o in glob.glob(os.path.join(B.OUT, "*.o")) if not o.endswith("_checked.o")]
    exe = tmp_path_factory.mktemp("probe") / "host_launches"
    # what the launch code does not call stays unresolved
    subprocess.run([B._nvcc(), *B.NVCC_FLAGS, "-cudart", "none", "-Xcompiler", "-no-pie", "-Xlinker",
                    "--unresolved-symbols=ignore-all", os.path.join(HERE, "_host_launches.cpp"), *objs,
                    "-o", str(exe)], check=True)

    def run(*args):
        return subprocess.run([str(exe), *map(str, args)], check=True, capture_output=True,
                              text=True).stdout.splitlines()
    return run


@pytest.mark.parametrize("priority", [0, -3])
def test_the_pass_over_the_packed_ranges_rest_never_starts_early(probe, priority):
    """It reads what the launch before it writes and does not wait for it."""
    for early in (1, 0):
        assert probe("launches", priority, early) == [
            f"tree early {early} priority {priority}", f"segmented early 0 priority {priority}",
            f"tree early {early} priority {priority}"]  # shared leaves: no second pass


def test_every_class_has_a_sum_tree_plan(probe):
    """Every cell size, model and number of cells, alone and behind the launches of
    other classes that fill the chip."""
    assert probe("plans") == []
