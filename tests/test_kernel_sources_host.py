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


def dependent_kernels():
    """{kernel: source file} of what is launched through launch_dependent."""
    found = {}
    for name in ("pg12.cu", "ntt.cu"):
        text = source(name)
        for call in re.findall(r"launch_dependent\(([^;]*);", text):
            for kernel in re.findall(r"\bk_\w+", call):
                found[kernel] = name
        if re.search(r"launch_dependent\(f,", text):
            found["k_ntt_pass"] = name
    return found


def test_dependent_launches_read_their_input_with_coherent_loads_after_the_wait():
    # a dependent launch is resident while the kernel before it writes: no load may
    # promise that nobody writes, and none may be moved above the wait
    kernels = dependent_kernels()
    assert {"k_tc_permute", "k_tc_sponge", "k_merkle_level", "k_merkle_top", "k_merkle_top_tail", "k_merkle_open",
            "k_merkle_verify_wide", "k_tc_verify", "k_ntt_pass", "k_ntt_bitrev"} <= set(kernels)
    for kernel, name in kernels.items():
        text = source(name)
        sig = re.search(r"\b%s\(([^)]*)\)\s*\{" % kernel, text).group(1)
        assert "__restrict__" not in sig, kernel
        code = body(text, kernel)
        wait = code.find("pdl_wait();")
        assert wait > 0, kernel
        assert not re.search(r"\b(ld1|ld2|ld1_cg|ld2_cg|load_words|load_chunk)\b", code[:wait]), kernel
    for name in ("pg12.cu", "ntt.cu", "tc_perm.cuh", "tcgen05.cuh", "poseidon.cuh"):
        text = source(name)
        assert "ld.global.nc" not in text and "__ldcg" not in text, name
        # only the constant tables, which no kernel writes
        assert "__ldg" not in text.replace(body(text, "load_consts"), "") if name == "poseidon.cuh" else "__ldg" not in text
    # the loads themselves are ordered against the wait
    for line in source("pg12.cu").splitlines():
        if re.search(r"\bld\.global\.(u64|v2|cg)", line):
            assert "volatile" in line and '"memory"' in line, line


def test_remote_shared_memory_is_written_only_once_its_block_has_started():
    # blocks of a cluster are scheduled together, but one may not have begun when
    # another stores into its shared memory: a cluster barrier comes first
    code = body(source("pg12.cu"), "k_merkle_top_tail")
    store = code.find("st.shared::cluster")
    first = code.find("barrier.cluster.wait")
    assert 0 <= code.find("barrier.cluster.arrive") < first < store
    # every block of the cluster takes that wait: no return or branch on the block comes before it
    assert "return" not in code[:first].split("auto build")[0] and "if (blockIdx" not in code[:first]
    # and a second barrier hands the stores over
    assert store < code.find("barrier.cluster.arrive", store) < code.find("barrier.cluster.wait", store)


def test_a_failed_tensor_core_kernel_waits_for_its_copies_before_it_ends():
    # after a wait has run out: one more bounded wait for the table copy and for the
    # last contraction, then the block meets and tensor memory is freed
    code = body(source("tc_perm.cuh"), "tc_teardown")
    failed = block(code, code.find("if (G.failed)"))
    assert "mbar_wait(reinterpret_cast<uint64_t *>(sm + L::kTabBar), 0)" in failed and "mbar_wait(G.mbar" in failed
    assert code.find(failed) < code.find("__syncthreads()") < code.find("tcgen05.dealloc")


def test_table_uploads_end_with_a_wait_for_the_copy():
    # a copy from pageable memory may return before the device holds the words
    for name, function in (("pg12.cu", "upload_tables"), ("pg12.cu", "pg_merkle_build_noalloc"),
                           ("ntt.cu", "ntt_upload_constants")):
        code = body(source(name), function)
        last = code.rfind("cudaMemcpyToSymbol")
        assert 0 <= last < code.find("cudaStreamSynchronize(cudaStreamLegacy)", last) < last + 160, function
