"""What the benchmark says runs: the kernel of a launch and its launches come from
the library's plan, not from the launch shape and the number of cells."""
import bench


def test_the_kernel_of_a_class_is_the_library_s_answer():
    c = {"V": 1024, "lanes_per_cell": 16, "warps_per_block": 2, "smem_layout": 1, "cells": 3000}
    assert bench.class_key(c, {"sum_tree": True}) == "V1024/tree"
    assert bench.class_key(c, {"sum_tree": False}) == "V1024/H16/rec/qb1/nd/u16"
    assert bench.chi_kernel_name("V1024/tree") == "k_chi_lane V1024/tree"
    assert bench.chi_kernel_name("V64/H8/pre/qb0/nd/u32").startswith("k_chi_seg ")
