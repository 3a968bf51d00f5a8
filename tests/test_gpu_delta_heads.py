"""The pass ahead of the backward kernel takes the heads of a token in groups of two passes, the next group's rows in flight: head
counts around a pass (two heads for D = 128, four for D = 64), a group, and the 64 heads whose statistics are fetched ahead."""
import pytest
import torch

from paper_2603_17484_b200 import l2a, synth
from tests.gpu_util import Case, check_backward_full, run_backward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Hq,Hkv,D", [(1, 1, 128), (3, 1, 128), (4, 2, 128), (5, 5, 128), (7, 1, 64), (9, 3, 64), (66, 11, 64)])
@pytest.mark.parametrize("flags", [0, l2a.FLAG_SHARED_WINDOW, l2a.FLAG_FORCE_ALL_GLOBAL], ids=["plain", "shared_window", "forced"])
def test_heads_around_a_group(Hq, Hkv, D, flags):
    B, L, W = 2, 150, 40
    d = synth.mask_bernoulli(B, L, 0.4, seed=Hq)
    c = Case(B, L, Hq, Hkv, D, W, d, seed=50 + Hq, backward=True, flags=flags)
    b = c.run_forward()
    run_backward(c)
    check_backward_full(c)
    # dgate_t = sum_h dO_t . a_t of the a_t that the forward stored, by compact row or, forced, by row
    dO, A = b.dO.double(), torch.zeros_like(b.dO, dtype=torch.float64)
    for i in range(B):
        if flags & l2a.FLAG_FORCE_ALL_GLOBAL:
            A[i] = b.A_c[i].double()
        else:
            n = int(b.n_routed[i])
            A[i, b.q_idx[i, :n].long()] = b.A_c[i, :n].double()
    want, size = (dO * A).sum(dim=(2, 3)), (dO * A).abs().sum(dim=(2, 3))
    # fp32: 8 sums in a lane, at most 4 shuffles, a sum per pass, 5 shuffles
    depth = 8 + 4 + -(-Hq * D // 256) + 5
    assert bool(((b.dgate.double() - want).abs() <= depth * 2.0 ** -24 * size).all())
