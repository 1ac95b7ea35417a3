"""Ordering rules of the kernels that no run on a GPU can be relied on to show.

Each check reads the kernel sources: a race or a missing wait gives the right
result almost every time, so the rule that excludes it is checked where it is
written.
"""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_09505_gb300", "csrc")


def source(name):
    """A kernel source without its comments."""
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


def block(text, start):
    """The parenthesised or braced text that opens at or after `start`, with its brackets."""
    i = min(k for k in (text.find("{", start), len(text)) if k >= 0)
    depth = 0
    for k in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[k], 0)
        if depth == 0:
            return text[i:k + 1]
    raise AssertionError("unbalanced braces")


def body(text, name):
    """The body of the function `name`."""
    return block(text, re.search(r"\b%s\([^;{]*\)\s*\{" % name, text).start())


def test_batch_kernel_raises_a_done_flag_only_after_its_group_has_met():
    # a root's words are stored by several warps; the thread that raises the flag
    # orders only its own stores and those a barrier has shown it
    text = source("pg12.cu")
    assert "signal_root" not in body(text, "k_tc_batch").replace("group_signal_root", "")
    helper = body(text, "group_signal_root")
    assert 0 <= helper.find("group_sync(") < helper.find("signal_root(")
