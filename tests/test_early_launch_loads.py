"""Kernels that may start before the kernel ahead of them has ended (they wait for it with
griddepcontrol.wait) read its results with plain loads only.  A load that the compiler may
treat as constant data, __ldg or one through a ``__restrict__`` pointer, can be moved ahead of
the wait and then races with the writes it is to follow."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2505_00315_gb300", "csrc")
FILES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))


def code_of(path):
    """The file without comments."""
    with open(path) as f:
        text = f.read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


def closing(text, at, pair):
    """Index just past the bracket that closes the one at ``at``."""
    depth = 0
    for i in range(at, len(text)):
        depth += (text[i] == pair[0]) - (text[i] == pair[1])
        if depth == 0:
            return i + 1
    raise AssertionError("unbalanced brackets")


def kernels(path):
    """(name, parameters, body) of every __global__ function."""
    text = code_of(path)
    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\s*(?=\())?", text):
        at = m.end()
        if text[at] == "(":   # the launch bounds
            at = closing(text, at, "()")
        name = re.match(r"\s*(\w+)\s*(?=\()", text[at:])
        start = at + name.end()
        end = closing(text, start, "()")
        body = text.index("{", end)
        yield name.group(1), text[start:end], text[body:closing(text, body, "{}")]


def test_the_kernels_are_found():
    found = {n: "griddepcontrol.wait" in b or "pdl_wait()" in b
             for p in FILES for n, _, b in kernels(p)}
    assert len(found) >= 20
    for name in ("dq_finish_kernel", "topk_select_kernel", "split_gemm_kernel", "rope_rows_kernel",
                 "attn_bwd_simt_kernel", "head_sum_kernel"):
        assert found[name], name
    assert not found["pad_wr_kernel"]


@pytest.mark.parametrize("path", FILES, ids=os.path.basename)
def test_waiting_kernels_use_plain_loads(path):
    assert "__ldg" not in code_of(path) and "ld.global.nc" not in code_of(path)
    for name, params, body in kernels(path):
        if "griddepcontrol.wait" in body or "pdl_wait()" in body:
            assert "__restrict__" not in params + body, name
