"""What the benchmark says runs: the kernel of a launch and its launches come from
the library's plan, not from the launch shape and the number of cells; the
sum-tree kernel's instructions per event are those of the current code."""
import bench


def test_the_kernel_of_a_class_is_the_library_s_answer():
    c = {"V": 1024, "lanes_per_cell": 16, "warps_per_block": 2, "smem_layout": 1, "cells": 3000}
    assert bench.class_key(c, {"sum_tree": True}) == "V1024/tree"
    assert bench.class_key(c, {"sum_tree": False}) == "V1024/H16/rec/qb1/nd/u16"
    assert bench.chi_kernel_name("V1024/tree") == "k_chi_lane V1024/tree"
    assert bench.chi_kernel_name("V64/H8/pre/qb0/nd/u32").startswith("k_chi_seg ")


def test_sum_tree_counts_were_measured_on_the_current_kernel():
    """A change of the kernel without a new measurement must fail here."""
    assert bench.TREE_IPE["sources"] == bench.chi_sources_sha(files=bench.TREE_SOURCES), (
        "the sum-tree chi kernel changed since its instructions per event were measured: "
        "re-run the ncu commands in profiles/k_chi_lane_inst_per_event.md")
    for key in ("batch:V1024", "batch:V256", "batch:V64", "medium:V256", "large:V1024"):
        ipe, bpe = bench.chi_ipe(*(key + "/tree").split(":"))
        assert 20 < ipe < 200 and 0 < bpe < 300


def test_the_sum_tree_hash_covers_every_file_of_the_kernel():
    import os
    import re
    seen, todo = set(), ["k_chi_lane.cu", "k_chi_lane_bind.cu", "k_chi_lane_pm.cu"]
    while todo:
        f = todo.pop()
        if f in seen:
            continue
        seen.add(f)
        with open(os.path.join(bench.CSRC, f)) as fh:
            todo += [x for x in re.findall(r'#include "(.*?)"', fh.read())
                     if os.path.exists(os.path.join(bench.CSRC, x))]
    # declarations only, and the wait for the launch before
    assert seen - set(bench.TREE_SOURCES) == {"tissue_internal.h", "early_launch.cuh"}
