"""Decode: chunks cut at the window's first key, whose partial results serve both modules, combined by the CTA that
finishes last.  Sizes around the cut and the chunk edges, against the fp64 oracle; repeated calls on one workspace."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_17484_b200 import l2a, synth
from tests.gpu_util import check_close, to_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Lk,Hq,Hkv,D,W", [
    (2, 1025, 2, 1, 128, 1023),      # one key before the window
    (2, 1025, 7, 1, 64, 1024),       # none
    (2, 257, 1, 1, 128, 0),          # a window of one key
    (3, 1281, 8, 2, 64, 255),        # whole chunks of 256 on both sides
    (5, 1300, 16, 4, 128, 300),      # ragged last chunks
    (1, 5000, 3, 3, 64, 4096),
    (3, 256, 14, 2, 128, 4096),      # a single chunk, routed or not
    (2, 400, 8, 1, 64, 128),         # a single chunk when not routed, two when routed
])
def test_chunks_around_the_window(B, Lk, Hq, Hkv, D, W):
    t = synth.qkv(B, 1, Hq, Hkv, D, seed=Lk + W, Lk=Lk)
    p = l2a.params(B, 1, Lk, Hq, Hkv, D, W)
    ws = torch.full((l2a.l2a_decode_workspace_bytes(p),), 0x5A, dtype=torch.uint8, device="cuda")   # nothing is expected in it
    q, K, V = (t[k].cuda() for k in ("Q", "K", "V"))
    sh = oracle.Shape(B, 1, Lk, Hq, Hkv, D, W)
    for d in (np.ones((B, 1), np.uint8), (np.arange(B) % 2).astype(np.uint8)[:, None], np.zeros((B, 1), np.uint8)):
        O = torch.full((B, 1, Hq, D), float("nan"), dtype=torch.bfloat16, device="cuda")
        l2a.l2a_decode(p, q, K, V, torch.from_numpy(d[:, 0].copy()).cuda(), O, ws)
        torch.cuda.synchronize()
        assert l2a.l2a_workspace_status(ws) == 0
        ref = oracle.forward_full(sh, synth.as_u16(t["Q"]), synth.as_u16(t["K"]), synth.as_u16(t["V"]), d)
        check_close(to_f64(O), ref["o"], "decode O")
        again = torch.empty_like(O)
        l2a.l2a_decode(p, q, K, V, torch.from_numpy(d[:, 0].copy()).cuda(), again, ws)
        assert torch.equal(O.view(torch.int16), again.view(torch.int16))      # fixed order, whichever CTA is last
