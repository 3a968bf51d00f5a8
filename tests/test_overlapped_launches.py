"""Kernels launched as programmatic dependents start while the kernel before them still runs.  What that one may still be
writing must not be read through the read-only path (`const __restrict__`, `__ldg`): such loads promise data that does
not change while the kernel runs, the time before its wait included, and may be moved above the wait."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_17484_b200", "csrc")
TEXT = "\n".join(re.sub(r"//[^\n]*", "", open(f).read()) for f in sorted(glob.glob(os.path.join(CSRC, "*.cu"))))


def kernel(name):
    """(parameters, body) of a __global__ function."""
    m = re.search(r"__global__[^;{]*?\b" + name + r"\s*\(", TEXT)
    assert m, name
    i, depth = m.end(), 1
    while depth:
        depth += {"(": 1, ")": -1}.get(TEXT[i], 0)
        i += 1
    params, j = TEXT[m.end():i - 1], TEXT.index("{", i)
    k, depth = j + 1, 1
    while depth:
        depth += {"{": 1, "}": -1}.get(TEXT[k], 0)
        k += 1
    return params, TEXT[j:k]


# inputs that a kernel ahead on the stream may still write when this one starts: for the gather that is whatever its caller
# launched last (the routing, the producer of the queries)
@pytest.mark.parametrize("name,inputs", [
    ("gather_rows_kernel", ["src", "q_idx", "n_routed", "prefix"]),
    ("dq_merge_kernel", ["acc_loc", "acc_glb"]),
    ("bwd_kernel", ["lse", "dl"]),
])
def test_no_read_only_loads_of_data_still_being_written(name, inputs):
    params, body = kernel(name)
    for x in inputs:
        assert not re.search(r"const[^,()]*\*\s*__restrict__\s+" + x + r"\b", params), x
        assert not re.search(r"__ldg\(\s*&?\s*" + x + r"\b", body), x
    if name != "bwd_kernel":
        assert "__ldg" not in body


def test_dependent_kernels_wait():
    names = set(re.findall(r"launch_dependent\(\s*(\w+)", TEXT)) - {"kern", "void"} | {"bwd_delta_kernel"}
    assert {"gather_rows_kernel", "attn_fwd_kernel", "bwd_kernel", "dq_merge_kernel", "route_scan_kernel"} <= names
    for n in names:
        assert "dependency_wait()" in kernel(n)[1], n
