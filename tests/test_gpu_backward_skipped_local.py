"""l2a_backward_split without the local part: the gradient of the local output takes no part, and is not read."""
import pytest
import torch

from paper_2603_17484_b200 import l2a, synth
from tests.gpu_util import Case, check_same_or_rounding, run_backward
from tests.test_overlapped_launches import kernel


def test_rows_of_a_skipped_local_part_are_those_of_the_other_gradient():
    """The pass ahead of the backward kernel asks for the rows of dO_loc in any case: they have to be dO's then."""
    _, body = kernel("bwd_delta_kernel")
    assert body.index("if (S == nullptr) dO_loc = dO;") < body.index("dO_loc + orow")
    assert body.count("dO_loc + ") == 1 and "__ldg(dO_loc" not in body and "dO_loc[" not in body


@pytest.mark.gpu
@pytest.mark.parametrize("B,L,Hq,Hkv,D", [(1, 300, 3, 1, 128), (2, 515, 8, 2, 64)])
def test_gradient_of_a_skipped_local_part_is_not_read(B, L, Hq, Hkv, D):
    d = synth.mask_bernoulli(B, L, 0.3, seed=L)
    c = Case(B, L, Hq, Hkv, D, 64, d, seed=9, backward=True)
    c.run_forward()
    b = c.buf
    c.p.flags |= l2a.FLAG_SKIP_LOCAL
    b.p.flags |= l2a.FLAG_SKIP_LOCAL
    want = [t.clone() for t in (run_backward(c).dQ, b.dK, b.dV, b.dgate)]
    unused = torch.empty(16, dtype=torch.uint8, device="cuda")
    for t in (b.dQ, b.dK, b.dV, b.dgate):
        t.fill_(float("nan"))
    l2a.l2a_backward_split(c.p, b.Q, b.K, b.V, b.d_mask, b.q_idx, b.n_routed, b.prefix, b.dO, unused, b.S_save, b.A_c,
                           b.lse_loc, b.lse_glb, b.dQ, b.dK, b.dV, b.dgate, b.bwd_ws)
    assert l2a.l2a_workspace_status(b.bwd_ws) == 0
    check_same_or_rounding(b.dQ, want[0], "dQ")
    for got, w in zip((b.dK, b.dV, b.dgate), want[1:]):
        assert torch.equal(got, w)
