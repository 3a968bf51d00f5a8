"""The fp32 dQ accumulators are cleared by the kernel of the row statistics up to 128 MiB of them and by one of their own beyond:
the backward over a workspace full of NaN, on both sides of that line and for the gradients of either module alone."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_17484_b200 import l2a, synth
from tests.gpu_util import Case, check_backward_full, check_close, run_backward, to_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,L,Hq,Hkv,D,W,rho", [
    (1, 1, 1, 1, 64, 4, 1.0),
    (1, 129, 2, 1, 128, 40, 0.4),
    (2, 700, 14, 2, 64, 100, 0.3),
    (1, 2040, 128, 64, 128, 16, 0.02),       # 127.5 MiB of rows
    (1, 2050, 128, 64, 128, 16, 0.02),       # 128.1 MiB
])
def test_backward_over_a_workspace_of_nan(B, L, Hq, Hkv, D, W, rho):
    c = Case(B, L, Hq, Hkv, D, W, synth.mask_bernoulli(B, L, rho, seed=3), seed=4, backward=True)
    c.run_forward()
    c.buf.bwd_ws.fill_(0xFF)
    run_backward(c)
    check_backward_full(c)


def test_either_module_alone():
    B, L, Hq, Hkv, D, W = 1, 500, 6, 2, 128, 60
    d = synth.mask_bernoulli(B, L, 0.3, seed=5)
    c = Case(B, L, Hq, Hkv, D, W, d, seed=6, backward=True)
    b = c.run_forward()
    u = [c.u16(k) for k in ("Q", "K", "V")]
    loc = oracle.backward_full(c.shape, *u, np.zeros_like(d), c.u16("dO"))
    both = oracle.backward_full(c.shape, *u, d, c.u16("dO"))
    for flag, want, args in ((l2a.FLAG_SKIP_GLOBAL, loc, (None, None, None, None)),
                             (l2a.FLAG_SKIP_LOCAL, [x - y for x, y in zip(both, loc)], (b.d_mask, b.q_idx, b.n_routed, b.prefix))):
        p = l2a.params(B, L, L, Hq, Hkv, D, W, flags=l2a.FLAG_SAVE_FOR_BWD | flag)
        b.bwd_ws.fill_(0xFF)
        l2a.l2a_backward(p, b.Q, b.K, b.V, *args, b.dO, b.S_save, b.A_c, b.lse_loc, b.lse_glb, b.dQ, b.dK, b.dV, None, b.bwd_ws)
        torch.cuda.synchronize()
        assert l2a.l2a_workspace_status(b.bwd_ws) == 0
        for got, x, name in zip((b.dQ, b.dK, b.dV), want, ("dQ", "dK", "dV")):
            check_close(to_f64(got), x, name + " of one module", outlier_frac=1e-5, early_rows=8)
