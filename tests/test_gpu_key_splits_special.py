"""Split key ranges and values that are not finite: what a routed row sees in one part reaches its result whatever the other parts
hold, what nobody wrote does not, and a part whose scores outweigh all others by far leaves the result of
that part alone."""
import numpy as np
import pytest
import torch

from tests.gpu_util import Case, split_plan

pytestmark = pytest.mark.gpu

LQ, LK, HQ, HKV, W = 60, 9000, 4, 2, 64
FAR = 5000                       # a key of a middle part, outside of every window, visible to every row


def _case(D, n=40):
    d = np.zeros((1, LQ), np.uint8)
    d[0, np.random.default_rng(2).permutation(LQ)[:n]] = 1
    c = Case(1, LQ, HQ, HKV, D, W, d, seed=21, Lk=LK, backward=True)
    c.buf.fwd_ws.fill_(0xFF)                                     # NaN in every slot
    return c, torch.from_numpy(d[0].astype(bool)).cuda()


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("tensor,value", [("K", "nan"), ("V", "nan"), ("V", "inf"), ("V", "-inf")])
def test_value_in_one_part(D, tensor, value):
    c, routed = _case(D)
    b = c.run_forward()
    assert split_plan(c, 1)[0][1] > 4
    clean, n = b.O.clone(), int(routed.sum())
    getattr(b, tensor)[0, FAR, 0, 5] = float(value)              # of the first KV head
    b.fwd_ws.fill_(0xFF)
    c.run_forward()
    hq = HQ // HKV
    assert torch.equal(b.O[0, ~routed], clean[0, ~routed])
    assert torch.equal(b.O[0, :, hq:], clean[0, :, hq:])         # the other KV head
    got = b.O[0, routed][:, :hq]
    if tensor == "K":
        assert got.isnan().all() and b.lse_glb[0, :hq, :n].isnan().all() and b.A_c[0, :n, :hq].isnan().all()
    else:
        hit = got[..., 5]
        assert (hit.isnan() if value == "nan" else hit == float(value)).all()
        rest = [i for i in range(D) if i != 5]
        assert torch.equal(got[..., rest], clean[0, routed][:, :hq][..., rest])
        assert b.lse_glb[0, :, :n].isfinite().all()
    assert b.lse_glb[0, hq:, :n].isfinite().all()


@pytest.mark.parametrize("D", [64, 128])
def test_one_part_outweighs_the_others(D):
    c, _ = _case(D)
    K = c.host["K"].clone()
    K[0, FAR:FAR + 3] *= 50                                      # scores of hundreds, both signs
    c.host["K"] = K
    c.buf.K.copy_(K)
    c.run_forward()
    ref = c.oracle_forward()
    n = int(c.d.sum())
    rows = np.nonzero(c.d[0])[0]
    got, want = c.buf.A_c[0, :n].double().cpu().numpy(), ref["a"][0, rows]
    assert np.isfinite(got).all()
    # fp32 sums of exact products put scores of some hundreds off by 1e-4, and so the probabilities: the bound of all outputs holds
    assert np.abs(got - want).max() <= 2e-2 + 2.0 ** -8 * np.abs(want).max()
