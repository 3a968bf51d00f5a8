"""Into how many parts the key ranges of the routed groups are split: both sides of the lines of that rule (seven and eight key
blocks; sixteen and seventeen; up to and beyond 32 groups; waves of equal groups), the most parts of a group, short prefills whose
groups differ in length, against the fp64 oracle."""
import numpy as np
import pytest
import torch

from paper_2603_17484_b200 import l2a
from tests.gpu_util import Case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Lq,Lk,Hq,Hkv,D,W,n_routed,flags", [
    (1, 30, 896, 2, 1, 128, 64, 9, 0),              # seven key blocks: none
    (1, 30, 897, 2, 1, 128, 64, 9, 0),              # eight: parts of two, the last block of a single key
    (1, 30, 2048, 2, 1, 64, 64, 9, 0),              # sixteen
    (1, 30, 2049, 2, 1, 64, 64, 9, 0),              # seventeen: by cost
    (1, 1100, 1100, 6, 1, 128, 100, 1100, 0),       # 26 groups of one to nine blocks, every token
    (33, 20, 1300, 1, 1, 64, 30, 11, 0),             # 33 groups: by cost
    (2, 300, 1100, 14, 2, 128, 50, 150, l2a.FLAG_SHARED_WINDOW),
    (1, 9, 20000, 1, 1, 128, 64, 5, 0),             # one group, the most parts
    (3, 64, 9000, 8, 8, 64, 200, 20, 0),            # 24 equal groups: one or two waves
])
def test_plan_of_key_splits(B, Lq, Lk, Hq, Hkv, D, W, n_routed, flags):
    d = np.zeros((B, Lq), np.uint8)
    rng = np.random.default_rng(5)
    for b in range(B):
        d[b, rng.permutation(Lq)[:max(1, n_routed - b % 3)]] = 1
    c = Case(B, Lq, Hq, Hkv, D, W, d, seed=18, Lk=Lk, flags=flags)
    if flags:
        c.buf.lse_loc = torch.empty(B, Hq, Lq, dtype=torch.float32, device="cuda")
    c.run_forward()
    c.check_forward_full()
    first = c.buf.O.clone()
    c.run_forward()                                 # the parts are combined in a fixed order
    assert torch.equal(first.view(torch.int16), c.buf.O.view(torch.int16))
