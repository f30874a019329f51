"""Kernels that may be resident while their predecessors still run (they call
grid_wait) read what those write through coherent loads: __ldg asks for data
that nobody writes during the kernel, so it may name a call's inputs only."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2608_23805_gb300", "csrc")
INPUTS = {"a.x", "a.wr", "a.wsg"}  # rows, router and shared-gate weights: written before the call


def kernels():
    """(name, body) of every __global__ function of the CUDA sources."""
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith(".cu"):
            continue
        with open(os.path.join(CSRC, f)) as fh:
            text = re.sub(r"//[^\n]*", "", fh.read())
        for m in re.finditer(r"__global__[^;{]*?(\w+_kernel)\(", text):
            start = text.index("{", m.end())
            depth, end = 1, start + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
            yield m.group(1), text[start:end]


def test_no_read_only_load_of_what_a_predecessor_writes():
    chained = {name: body for name, body in kernels() if "grid_wait()" in body}
    assert {"combine_kernel", "fused_cols_kernel", "scatter_kernel", "router_select_kernel"} <= set(chained)
    for name, body in chained.items():
        for m in re.finditer(r"__ldg\(", body):
            arg = body[m.end():m.end() + 120]
            named = re.findall(r"\ba\.\w+|\bperm\b", arg)
            assert named and named[0] in INPUTS, f"{name}: __ldg({arg.split(';')[0]}"
