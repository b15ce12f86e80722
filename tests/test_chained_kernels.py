"""Kernels launched while the one before them runs (lbrr_chain.cuh) take their
memory by plain pointers.

What the kernel before wrote may be read only after chain_wait(). For a
__restrict__ parameter the language lets a compiler move the loads ahead of that
statement, so no such kernel has one.
"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1505_06900_gb300", "csrc")


def _kernels(text):
    """(name, parameters, body) of the __global__ functions of a source file."""
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"__global__\s+void\b", text):
        head = re.compile(r"(?:__launch_bounds__\([^;{]*?\)\s*)?(\w+)\(([^{}]*)\)\s*\{").search(
            text, m.end())
        depth, end = 1, head.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[end], 0)
            end += 1
        yield head.group(1), head.group(2), text[head.end():end]


def test_no_restrict_parameter_is_read_after_the_wait():
    chained = {}
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        for name, params, body in _kernels(open(path).read()):
            if "chain_wait()" in body:
                chained[name] = params
    assert {"rr_step_walls_kernel", "rr_moment_pass2_kernel", "rr_moment_march_kernel",
            "mlp_conv_kernel", "feature_source_kernel", "mlp_train_tc_kernel",
            "mlp_reduce_adam_kernel"} <= set(chained)
    assert [n for n, p in chained.items() if "__restrict__" in p] == []
