"""A call that uses every slot of the forward workspace of its shape: nothing is written behind it."""
import numpy as np
import pytest

from paper_2603_17484_b200 import l2a
from tests.gpu_util import Case, split_plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Lq,Lk,Hq,Hkv,D,groups", [(1, 9, 120000, 1, 1, 64, 1), (2, 30, 100000, 16, 2, 128, 4)])
def test_every_slot_in_use(B, Lq, Lk, Hq, Hkv, D, groups):
    c = Case(B, Lq, Hq, Hkv, D, 64, np.ones((B, Lq), np.uint8), seed=2, Lk=Lk, flags=l2a.FLAG_SKIP_LOCAL)
    assert c.buf.fwd_ws.numel() <= 32 * groups * 256 * (D + 2) * 4 + 1024
    c.run_forward()                                        # (checks the guards around every buffer)
    assert split_plan(c, groups) == [(32, 32)] * groups
