"""Orders inside kernels that no run can show to be right: read from the source."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2402_05109_b200", "csrc")


def kernel_bodies(name):
    """Every kernel's text, from its __global__ to the closing brace in the first column."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    return [text[m.start():text.index("\n}", m.start())] for m in re.finditer(r"^__global__", text, re.M)]


def test_a_cluster_has_started_before_its_shared_memory_is_stored_to():
    """Distributed shared memory may be accessed once every CTA of the cluster is known to run: a cluster barrier completes first."""
    found = 0
    for body in kernel_bodies("kernels.cu"):
        if "st.shared::cluster" in body:
            found += 1
            assert -1 < body.find("barrier.cluster.arrive") < body.find("barrier.cluster.wait") < body.find("st.shared::cluster")
    assert found == 1


def test_only_weights_and_tables_are_declared_constant():
    """`const ... __restrict__` lets the compiler move loads over the dependency wait, which is right for data that no kernel writes."""
    constant = set()
    for body in kernel_bodies("kernels.cu"):
        constant |= set(re.findall(r"const \w+\s*\*\s*__restrict__\s+(\w+)", body[:body.index("{")]))
    assert constant <= {"embed", "gain", "bias", "first_child", "n_child", "path_tab"}


def test_gemm_operands_are_whole_buffers():
    """The tensor-core GEMM reads row tiles of up to 15 rows more than it is asked for, as far as the buffer that it is told of goes: operand and row
    count of a call are those of one buffer of the workspace, and rows inside it are named by their number."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "hydra.cu")).read())
    carved = dict(re.findall(r"auto\* (\w+) = b\.take<char>\(\(size_t\)np \* (\w+) \*", text))
    assert {"xn", "attn_out", "act", "z", "yb"} <= set(carved)
    calls = re.findall(r"run_gemm\(c, ([^,]+), ([^,]+),", text)
    assert len(calls) >= 10
    for x, rows in calls:
        assert x.startswith("c->") and rows == "c->" + carved[x[3:]], (x, rows)
