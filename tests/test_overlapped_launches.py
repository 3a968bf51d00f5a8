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
    ("gather_rows_kernel", ["src", "src2", "q_idx", "n_routed"]),
    ("attn_fwd_kernel", []),                  # queries and routing, which the arguments hold: no read-only load at all
    ("fwd_combine_kernel", []),
    ("dq_merge_kernel", ["acc_loc", "acc_glb"]),
    ("bwd_kernel", ["lse", "dl"]),
])
def test_no_read_only_loads_of_data_still_being_written(name, inputs):
    params, body = kernel(name)
    if name in ("gather_rows_kernel", "dq_merge_kernel"):
        assert all(re.search(r"\*\s*(?:__restrict__\s+)?" + x + r"\b", params) for x in inputs), params
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


# Kernels that touch memory ahead of their wait, and why they may: Delta reads nothing that the gather ahead of it writes (below);
# the global pass overlaps with the local one alone, which is a plain launch and writes only what is read behind the wait.
LATE = {"bwd_delta_kernel", "attn_fwd_kernel"}


def test_all_other_kernels_touch_no_memory_ahead_of_their_wait():
    names = set(re.findall(r"launch_dependent\(\s*(\w+)", TEXT)) - {"kern", "void"} - LATE
    assert {"attn_fwd_local_kernel", "decode_combine_kernel", "bwd_kernel", "dq_zero_kernel", "dq_merge_kernel"} <= names
    for n in names:
        params, body = kernel(n)
        ahead = body[:body.index("dependency_wait()")]
        pointers = re.findall(r"\*\s*(?:__restrict__\s+)?(\w+)\s*(?:,|$)", params)
        structs = re.findall(r"\b\w+Args\s*&?\s*(\w+)", params)
        assert pointers or structs, n
        for x in pointers:
            assert not re.search(r"\b" + x + r"\b", ahead), (n, x)
        for x in structs:
            assert not re.search(r"\b" + x + r"\.\w+\s*\[|[=(,]\s*[*&]\s*" + x + r"\.\w+", ahead), n
            assert "make_" not in ahead and "_at(" not in ahead, n


def arguments(call, text):
    """Top-level arguments of the first call in the text."""
    i = text.index(call) + len(call)
    out, depth, start = [], 1, i
    while depth:
        c = text[i]
        depth += {"(": 1, "{": 1, "[": 1, ")": -1, "}": -1, "]": -1}.get(c, 0)
        if depth == 0 or (depth == 1 and c == ","):
            out.append(" ".join(text[start:i].split()))
            start = i + 1
        i += 1
    return out


def test_delta_reads_nothing_that_the_gather_ahead_of_it_writes():
    backward = TEXT[TEXT.rindex("static l2a_status backward_impl("):]
    declared = open(os.path.join(CSRC, "l2a_common.cuh")).read()
    formal = arguments("cudaError_t launch_gather_rows(", re.sub(r"//[^\n]*", "", declared))
    gather = arguments("launch_gather_rows(", backward)
    arg = {re.sub(r"\s*=.*", "", f).split()[-1].lstrip("*"): g for f, g in zip(formal, gather)}
    assert arg["overlap"] == "false"             # everything before it has completed when Delta starts
    written = [re.search(r"\w+\)?$", arg[k]).group().rstrip(")") for k in ("dst", "dst2")]
    assert written == ["Qc", "dOc"] and re.search(r"\(ws\)", arg["zero"])      # beside the header of the workspace
    delta = arguments("launch_dependent(kern,", backward)
    for a in delta:
        assert not re.search(r"\b(" + "|".join(written) + r"|ws)\b", a), a
    read = {"src": "Q", "q_idx": "q_idx", "n_routed": "n_routed", "src2": "dO"}
    for k, v in read.items():                    # and the gather reads nothing that Delta writes
        assert re.search(r"\b" + v + r"\b", arg[k]), k
    _, body = kernel("bwd_delta_kernel")
    stores = set(re.findall(r"\b(\w+)\[[^\];]*\]\s*=[^=]", body))
    assert {"delta_loc", "delta_glb", "lse_eff", "dgate"} <= stores and not stores & {"dO", "S", "A_c", "prefix", "d_mask"}
