"""Global Attention with split key ranges (few routed groups over many keys): the combination of the parts against the
fp64 oracle, for every kind of launch that reaches it, and the rule that the host-buffer step gives the same bits.  Every case says
into how many parts its longest group is split, and fails if the plan is another one."""
import numpy as np
import pytest
import torch

from paper_2603_17484_b200 import l2a, synth
from tests.gpu_util import Case, check_backward_full, check_close, run_backward, split_plan, to_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lq,Lk,Hq,Hkv,D,W,n_routed,flags,backward,parts", [
    (40, 4096, 2, 1, 128, 64, 5, 0, False, 11),        # 32 blocks
    (40, 4095, 2, 1, 64, 64, 40, 0, False, 11),        # ragged last block
    (300, 6200, 1, 1, 128, 100, 300, 0, True, 17),     # two groups, a ragged second one; 49 blocks
    (513, 16700, 2, 1, 64, 128, 290, 0, False, 27),    # the second tile of the second group empty
    (200, 5000, 2, 2, 128, 2200, 150, l2a.FLAG_SHARED_WINDOW, False, 1),    # 22 blocks before the window: undivided
    (200, 6000, 2, 2, 128, 700, 150, l2a.FLAG_SHARED_WINDOW, False, 6),     # keys before the window only: 42 blocks at most
    (300, 7000, 6, 2, 64, 1500, 200, l2a.FLAG_SHARED_WINDOW, True, 4),      # packed heads
    (200, 9000, 2, 1, 64, 300, 60, l2a.FLAG_SHARED_WINDOW, True, 14),
    (600, 5000, 64, 8, 64, 64, 12, 0, False, 10),      # equal groups behind a local pass of 192 items
])
def test_split_key_ranges(Lq, Lk, Hq, Hkv, D, W, n_routed, flags, backward, parts):
    d = np.zeros((1, Lq), np.uint8)
    d[0, np.random.default_rng(3).permutation(Lq)[:n_routed]] = 1
    c = Case(1, Lq, Hq, Hkv, D, W, d, seed=8, Lk=Lk, backward=backward, flags=flags)
    if flags and not backward:
        c.buf.lse_loc = torch.empty(1, Hq, Lq, dtype=torch.float32, device="cuda")
    c.run_forward()
    c.check_forward_full()
    assert split_plan(c, 1) == [(parts, parts)]
    first = c.buf.O.clone()
    c.run_forward()                                # the parts are combined in a fixed order
    assert torch.equal(first.view(torch.int16), c.buf.O.view(torch.int16))
    if backward:
        run_backward(c)
        check_backward_full(c)


def test_batch_entries_of_different_routed_counts():
    d = np.zeros((3, 300), np.uint8)
    d[0, ::3] = 1
    d[2, 7] = 1                                    # entry 1 has none
    c = Case(3, 300, 2, 1, 64, 50, d, seed=9, Lk=6000)
    c.run_forward()
    assert split_plan(c, 1) == [(16, 16)]
    c.check_forward_full()


def test_global_part_alone():
    """Without a local pass in the call: routed rows hold the global result, all others zeros."""
    d = np.zeros((1, 100), np.uint8)
    d[0, ::4] = 1
    c = Case(1, 100, 8, 4, 64, 100, d, seed=10, Lk=8000, flags=l2a.FLAG_SKIP_LOCAL)
    c.run_forward()
    assert split_plan(c, 1) == [(21, 21)]
    rows = np.nonzero(d[0])[0]
    out = to_f64(c.buf.O)[0]
    check_close(out[rows], c.oracle_forward()["a"][0, rows], "O of the global part alone")
    assert not out[d[0] == 0].any()


def test_host_step_in_row_ranges_gives_the_same_bits():
    B, L, Hq, Hkv, D, W = 1, 8192 + 100, 2, 1, 64, 128
    d = synth.mask_bernoulli(B, L, 0.05, seed=4)
    c = Case(B, L, Hq, Hkv, D, W, d, seed=11)
    c.run_forward()
    want = c.buf.O.clone()
    host = {k: v.pin_memory() for k, v in c.host.items()}
    host["router"] = torch.from_numpy(d).pin_memory()
    host["O"] = torch.empty_like(want, device="cpu").pin_memory()
    c.buf.O.zero_()
    l2a.l2a_step_host(c.p, host, c.buf, l2a.ROUTER_MASK_U8, 0.0)
    assert torch.equal(host["O"].view(torch.int16), want.cpu().view(torch.int16))
