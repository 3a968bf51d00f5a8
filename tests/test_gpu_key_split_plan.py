"""Into how many parts the key ranges of the routed groups are split, on either side of where the rule changes: calls of fewer than
32 key blocks (never), few and many groups, one group with the most parts, waves of equal groups, short prefills whose groups differ
in length -- against the fp64 oracle."""
import numpy as np
import pytest
import torch

from paper_2603_17484_b200 import l2a
from tests.gpu_util import Case, split_plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Lq,Lk,Hq,Hkv,D,W,n_routed,flags,slots", [
    (1, 30, 896, 2, 1, 128, 64, 9, 0, 1),              # fewer than 32 key blocks
    (1, 30, 897, 2, 1, 128, 64, 9, 0, 1),
    (1, 30, 2048, 2, 1, 64, 64, 9, 0, 1),
    (1, 30, 2049, 2, 1, 64, 64, 9, 0, 1),
    (1, 1100, 1100, 6, 1, 128, 100, 1100, 0, 1),       # 26 groups of one to nine blocks, every token
    (33, 20, 1300, 1, 1, 64, 30, 11, 0, 1),
    (2, 300, 1100, 14, 2, 128, 50, 150, l2a.FLAG_SHARED_WINDOW, 1),
    (1, 9, 20000, 1, 1, 128, 64, 5, 0, 32),            # one group, the most parts
    (3, 64, 9000, 8, 8, 64, 200, 20, 0, 5),            # 24 equal groups: waves on the SMs that the local pass leaves and on its own
    (40, 20, 4300, 1, 1, 64, 30, 11, 0, 2),            # 40 of 34 blocks
    (1, 4300, 4300, 4, 2, 64, 100, 900, 0, 7),         # a prefill: 16 groups of two to 34 blocks
])
def test_plan_of_key_splits(B, Lq, Lk, Hq, Hkv, D, W, n_routed, flags, slots):
    d = np.zeros((B, Lq), np.uint8)
    rng = np.random.default_rng(5)
    for b in range(B):
        d[b, rng.permutation(Lq)[:max(1, n_routed - b % 3)]] = 1
    c = Case(B, Lq, Hq, Hkv, D, W, d, seed=18, Lk=Lk, flags=flags)
    if flags:
        c.buf.lse_loc = torch.empty(B, Hq, Lq, dtype=torch.float32, device="cuda")
    c.run_forward()
    assert split_plan(c, 1)[0][0] == slots, split_plan(c, 1)
    c.check_forward_full()
    first = c.buf.O.clone()
    c.run_forward()                                 # the parts are combined in a fixed order
    assert torch.equal(first.view(torch.int16), c.buf.O.view(torch.int16))
