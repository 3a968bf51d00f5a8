"""Routing and compaction around the block edges: sequences of one to four blocks of 4096 positions take one launch, longer
ones two; results are exact."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_17484_b200 import l2a

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [1, 31, 33, 511, 513, 4095, 4096, 4097, 16384, 16385, 40001])
@pytest.mark.parametrize("kind", [l2a.ROUTER_MASK_U8, l2a.ROUTER_LOGITS_F32, l2a.ROUTER_LOGITS_BF16])
def test_block_edges(L, kind):
    B = 3
    rng = np.random.default_rng(L)
    d = (rng.random((B, L)) < np.array([[0.0], [0.4], [1.0]])).astype(np.uint8)
    p = l2a.params(B, L, L, 1, 1, 64, 8)
    if kind == l2a.ROUTER_MASK_U8:
        router = torch.from_numpy(d * rng.integers(1, 255, d.shape).astype(np.uint8)).cuda()
    else:
        z = np.where(d == 1, rng.random(d.shape), -0.01 - rng.random(d.shape)).astype(np.float32)
        router = torch.from_numpy(z).cuda().to(torch.float32 if kind == l2a.ROUTER_LOGITS_F32 else torch.bfloat16)
    dm = torch.full((B, L), 9, dtype=torch.uint8, device="cuda")
    qi = torch.full((B, L), 9, dtype=torch.int32, device="cuda")
    n = torch.full((B,), 9, dtype=torch.int32, device="cuda")
    pf = torch.full((B, L + 1), 9, dtype=torch.int32, device="cuda")
    ws = torch.full((l2a.l2a_workspace_bytes(p)[0],), 0xFF, dtype=torch.uint8, device="cuda")
    l2a.l2a_route_compact(p, router, kind, 0.0, dm, qi, n, pf, ws)
    torch.cuda.synchronize()
    assert l2a.l2a_workspace_status(ws) == 0
    q_idx, cnt, prefix = oracle.compact(d)
    assert np.array_equal(dm.cpu().numpy(), d)
    assert np.array_equal(n.cpu().numpy(), cnt) and np.array_equal(pf.cpu().numpy(), prefix)
    assert np.array_equal(qi.cpu().numpy(), q_idx)
