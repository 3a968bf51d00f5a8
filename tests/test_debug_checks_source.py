"""The index-checking build: an index into the queries is checked before the kernel that gathers them forms an address from it."""
import re

import pytest

from tests.test_overlapped_launches import kernel


@pytest.mark.parametrize("name,address,check", [
    ("attn_fwd_kernel", "a.q_st.t", r"dbg_in_range\(t >= 0 && t < a\.Lq, a\.status\)"),
    ("gather_rows_kernel", "t * src_row_chunks", r"dbg_in_range\(t >= 0 && t < L, status\)"),
])
def test_index_is_checked_before_the_address(name, address, check):
    body = kernel(name)[1]
    assert re.search(check, body[:body.index(address)]), name
