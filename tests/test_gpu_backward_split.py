"""Backward with one, two and four CTAs per key block (l2a picks by the number of key blocks x KV heads x batch against
the number of SMs: 148 on the device these sizes are chosen for), against the fp64 oracle."""
import pytest

from paper_2603_17484_b200 import synth
from tests.gpu_util import Case, check_backward_full, run_backward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,L,Lk,Hq,Hkv,D,W,rho", [
    (1, 100, 100, 1, 1, 128, 64, 0.0),       # one item: three of the four CTAs have none
    (1, 100, 100, 2, 1, 64, 64, 0.5),        # two to four items
    (1, 90, 400, 3, 1, 128, 17, 0.3),        # key blocks that no query sees
    (1, 1000, 1000, 7, 1, 128, 300, 0.4),    # 8 blocks: four CTAs
    (2, 515, 515, 8, 8, 128, 200, 0.3),      # 80 blocks: two
    (1, 1280, 1280, 20, 20, 64, 128, 0.2),   # 200 blocks: two
    (2, 1000, 1000, 14, 14, 64, 250, 0.2),   # 224 blocks: one
])
def test_backward_split(B, L, Lk, Hq, Hkv, D, W, rho):
    d = synth.mask_bernoulli(B, L, rho, seed=5)
    c = Case(B, L, Hq, Hkv, D, W, d, seed=6, Lk=Lk, backward=True)
    c.run_forward()
    run_backward(c)
    check_backward_full(c)
