"""The multiply results bench.py says a kernel executes, checked on the CPU."""
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

import bench  # noqa: E402


def test_tensor_core_kernels_execute_no_linear_layer():
    # 118 S-boxes of four products and 90 chain products, 8 results each; a node
    # or a first chunk skips four S-boxes
    assert bench.executed_mul32_per_perm("k_tc_permute", 1) == 118 * 32 + 90 * 8 == 4496
    assert bench.executed_mul32_per_perm("k_tc_sponge:level", 8) == 114 * 32 + 90 * 8
    assert bench.executed_mul32_per_perm("k_tc_sponge:leaves", 8) == 4496 - 128 / 8
    assert bench.executed_mul32_per_perm("k_tc_sponge:leaves", 1, small=True) == 4496 - 128


def test_integer_kernels_execute_the_method_less_what_they_skip():
    assert bench.executed_mul32_per_perm("k_permute", 1) == bench.MUL_RESULTS_PER_PERM
    assert bench.executed_mul32_per_perm("k_merkle_level", 4) == 16568 - (4 * 28 + 48 * 8) - 96 * 8
    assert bench.executed_mul32_per_perm("k_merkle", 1, small=True) == 12536 - (4 * 28 + 48 * 4) - 96 * 4


def test_forms_whose_lanes_repeat_work_are_not_counted():
    for kernel in ("k_merkle_top", "k_merkle_top_leaf", "k_merkle_top_tail", "k_batch_top", "k_ntt_pass"):
        assert bench.executed_mul32_per_perm(kernel, 1) is None
