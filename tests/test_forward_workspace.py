"""Size of the forward workspace: the slots that the parts of split key ranges can take, or one copy of Q if that is more.  It follows
from queries, heads and batch alone, so that a workspace serves every chunk of a prompt, and grows with each of them."""
import pytest

from paper_2603_17484_b200 import build as l2a_build
from paper_2603_17484_b200 import l2a


def size(B, Lq, Hq, Hkv, D, Lk=None, W=128, **kw):
    return l2a.l2a_workspace_bytes(l2a.params(B, Lq, Lk or Lq, Hq, Hkv, D, W, **kw))[1]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    l2a_build.build_lib()


@pytest.mark.parametrize("B,Lq,Hq,Hkv,D", [
    (1, 131072, 32, 8, 128), (1, 2000, 32, 8, 128), (1, 64, 28, 4, 128), (1, 1, 1, 1, 64), (1, 9, 8, 1, 64), (3, 300, 12, 2, 64), (2, 4096, 28, 4, 128),
])
def test_size_is_that_of_the_slots(B, Lq, Hq, Hkv, D):
    groups = -(-Lq * (Hq // Hkv) // 256) * Hkv * B
    slots = min(4 * 148, 32 * min(groups, 128))            # parts of all groups, parts of a group
    want = max(slots * 256 * (D + 2) * 4, B * Lq * Hq * D * 2)
    assert want <= size(B, Lq, Hq, Hkv, D) <= want + 1024


def test_size_serves_other_calls():
    ref = size(1, 2000, 28, 4, 128)
    for kw in (dict(Lk=2000), dict(Lk=34000), dict(Lk=120000, W=4096), dict(Lk=5000, q_pos_offset=0)):
        assert size(1, 2000, 28, 4, 128, **kw) == ref
    last = 0
    for Lq in list(range(1, 700, 13)) + [1000, 5000, 40000]:
        n = size(1, Lq, 12, 2, 64)
        assert n >= last
        last = n
        assert size(2, Lq, 12, 2, 64) >= n and size(1, Lq, 6, 1, 64) <= n
