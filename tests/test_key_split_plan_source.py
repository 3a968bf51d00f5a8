"""The plan of key splits is a comparison of costs in fp32.  One kernel makes it and leaves it in the workspace; the kernel that
combines the parts must not make it again, since another compilation may contract or round the same expressions differently."""
import re

from tests.test_overlapped_launches import TEXT, kernel


def test_only_the_attention_kernel_makes_the_plan():
    assert len(re.findall(r"\bkey_split\(", TEXT)) == 2          # the function and one call
    assert "key_split(" in kernel("attn_fwd_kernel")[1]
    body = kernel("fwd_combine_kernel")[1]
    assert "key_split(" not in body and "group_parts[" in body
