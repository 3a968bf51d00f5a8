"""Key ranges of fewer than 32 blocks of 128 keys are not split, whatever the call: routed rows of such a sequence have the same bits
alone, in a batch of any size and as a head shard.  From 32 blocks on the parts follow from the whole call."""
import numpy as np
import pytest
import torch

from paper_2603_17484_b200 import l2a
from tests.gpu_util import Case, split_plan

pytestmark = pytest.mark.gpu

OUT = ("O", "A_c", "lse_loc", "lse_glb")


def _mask(L, n, seed):
    d = np.zeros((1, L), np.uint8)
    d[0, np.random.default_rng(seed).permutation(L)[:n]] = 1
    return d


def _rows(buf, b, n, what):
    t = getattr(buf, what)
    if what == "O":
        return t[b]
    return t[b, :n] if what == "A_c" else t[b, :, :n] if what == "lse_glb" else t[b]


@pytest.mark.parametrize("Lq,Lk,Hq,Hkv,D,W,n,flags", [
    (1024, 1024, 4, 2, 128, 128, 200, 0),                # 8 blocks
    (2177, 2177, 8, 2, 64, 100, 400, 0),                 # 18
    (3000, 3000, 4, 4, 128, 4096, 300, 0),               # 24
    (64, 3968, 8, 4, 128, 128, 20, 0),                   # 31, a few new tokens
    (300, 3900, 4, 2, 64, 200, 60, l2a.FLAG_SHARED_WINDOW),
])
def test_alone_in_a_batch_and_as_a_shard(Lq, Lk, Hq, Hkv, D, W, n, flags):
    B = 5
    d = np.concatenate([_mask(Lq, max(1, n - 7 * b), b) for b in range(B)])
    batch = Case(B, Lq, Hq, Hkv, D, W, d, seed=3, Lk=Lk, flags=flags | l2a.FLAG_SAVE_FOR_BWD, backward=True)
    batch.run_forward()
    for b in (0, 3):
        c = Case(1, Lq, Hq, Hkv, D, W, d[b:b + 1], seed=3, Lk=Lk, flags=flags, backward=True)
        for k in ("Q", "K", "V"):
            getattr(c.buf, k).copy_(getattr(batch.buf, k)[b:b + 1])
        c.run_forward()
        for k in OUT:
            got, want = _rows(c.buf, 0, int(d[b].sum()), k), _rows(batch.buf, b, int(d[b].sum()), k)
            assert torch.equal(got, want), (b, k)
        # one KV head of it
        hq = Hq // Hkv
        s = Case(1, Lq, hq, 1, D, W, d[b:b + 1], seed=3, Lk=Lk, flags=flags, backward=True)
        for k, h in (("Q", hq), ("K", 1), ("V", 1)):
            getattr(s.buf, k).copy_(getattr(c.buf, k)[:, :, -h:])
        s.run_forward()
        assert torch.equal(s.buf.O, c.buf.O[:, :, -hq:]), b
    assert split_plan(batch, 1) == [(1, 1)]


def test_line_at_32_blocks():
    for Lk, split in ((3968, False), (3969, True)):      # 31 and 32 blocks
        c = Case(1, 40, 2, 1, 128, 64, _mask(40, 9, 1), seed=4, Lk=Lk)
        c.run_forward()
        (slots, parts), = split_plan(c, 1)
        assert (slots > 1) == split and (parts > 1) == split, (Lk, slots, parts)
        c.check_forward_full()


@pytest.mark.parametrize("last,split", [(895, False), (896, True)])      # in the seventh and in the eighth block
def test_short_group_of_a_longer_call(last, split):
    d = np.zeros((1, 5000), np.uint8)
    d[0, last - 255:last + 1] = 1
    d[0, 4700:4956] = 1                                  # the other group, of 39 blocks: split
    c = Case(1, 5000, 1, 1, 128, 64, d, seed=6)
    c.run_forward()
    plan = split_plan(c, 2)
    assert plan[0][1] > 1 and (plan[1][1] > 1) == split, plan
    c.check_forward_full()
