"""The global pass leaves the plan of its key splits in the workspace, for every group of the launch, undivided ones included; the
combination has no other source for it."""
import numpy as np
import pytest

from paper_2603_17484_b200 import l2a
from tests.gpu_util import Case, split_plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Lq,Lk,Hq,Hkv,D,W,n_routed,groups,most", [
    (1, 40, 9000, 2, 1, 128, 64, 9, 1, 32),            # one group in many parts
    (2, 600, 9000, 4, 2, 64, 64, 300, 12, 32),         # three groups a KV head
    (1, 4500, 4500, 2, 2, 128, 100, 1000, 8, 32),      # the first group's rows see fewer key blocks than the last one's
    (1, 40, 600, 2, 1, 128, 64, 9, 1, 1),              # five key blocks: undivided
])
def test_plan_is_stored(B, Lq, Lk, Hq, Hkv, D, W, n_routed, groups, most):
    d = np.zeros((B, Lq), np.uint8)
    for b in range(B):
        d[b, np.random.default_rng(b).permutation(Lq)[:n_routed]] = 1
    c = Case(B, Lq, Hq, Hkv, D, W, d, seed=5, Lk=Lk)
    c.buf.fwd_ws.fill_(0x55)
    c.run_forward()
    plan = split_plan(c, groups)
    slots = plan[0][0]
    assert 1 <= slots <= most and (most == 1) == (slots == 1), plan
    for s, n in plan:
        assert s == slots and 1 <= n <= slots, plan
    assert most == 1 or plan[0][1] > 1, plan
    c.check_forward_full()


@pytest.mark.parametrize("B,Lq,Lk,Hq,Hkv,D,W,n_routed,flags,slots", [
    (1, 4096, 4096, 4, 4, 64, 4096, 819, 0, 1),          # 16 groups that end under the local pass, which leaves them SMs
    (1, 8192, 8192, 1, 1, 64, 4096, 410, 0, 2),          # two groups, longer than the local pass's items
    (1, 20000, 20000, 1, 1, 64, 4096, 2000, 0, 5),
    (1, 4096, 4096, 4, 4, 64, 128, 819, 0, 8),           # a local pass that is over early
    (1, 2000, 34000, 32, 8, 64, 4096, 600, 0, 3),        # 80 equal groups behind a local pass of 256 items
    (1, 100, 8000, 8, 4, 64, 100, 60, l2a.FLAG_SKIP_LOCAL, 21),   # no local pass: one wave of equal items
    (1, 100, 8000, 8, 4, 64, 4096, 60, 0, 2),            # the same beside one of eight long items
])
def test_plan_follows_the_local_pass(B, Lq, Lk, Hq, Hkv, D, W, n_routed, flags, slots):
    d = np.zeros((B, Lq), np.uint8)
    d[0, np.random.default_rng(7).permutation(Lq)[:n_routed]] = 1
    c = Case(B, Lq, Hq, Hkv, D, W, d, seed=5, Lk=Lk, flags=flags)
    c.run_forward()
    assert split_plan(c, 1)[0][0] == slots, split_plan(c, 1)
