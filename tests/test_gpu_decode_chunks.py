"""Decode: chunks cut at the window's first key, whose partial results serve both modules, combined by a kernel behind
them.  Sizes around the cut and the chunk edges, against the fp64 oracle; repeated calls on one workspace."""
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


@pytest.mark.parametrize("B,Lk,Hq,Hkv,D,W", [
    (2, 9001, 28, 4, 128, 4096),     # half of a routed token's cache is its window
    (4, 6000, 32, 8, 64, 4096),
    (3, 20000, 8, 1, 128, 1000),
    (2, 300, 12, 2, 128, 4096),      # one chunk, which is window and whole cache
])
def test_error_is_that_of_rounding_the_result(B, Lk, Hq, Hkv, D, W):
    """Against 64 bits, in the 2-norm: what rounding the exact result to bf16 costs, and no more than 2 % beside it (scores and
    sums in fp32; what P loses in bf16 has its own rows of the product).  With P in bf16 alone it was 1.2 to 1.3 times that."""
    t = synth.qkv(B, 1, Hq, Hkv, D, seed=Lk, Lk=Lk)
    d = np.ones((B, 1), np.uint8)
    p = l2a.params(B, 1, Lk, Hq, Hkv, D, W)
    ws = torch.empty(l2a.l2a_decode_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    O = torch.empty((B, 1, Hq, D), dtype=torch.bfloat16, device="cuda")
    l2a.l2a_decode(p, t["Q"].cuda(), t["K"].cuda(), t["V"].cuda(), torch.from_numpy(d[:, 0].copy()).cuda(), O, ws)
    sh = oracle.Shape(B, 1, Lk, Hq, Hkv, D, W)
    want = oracle.forward_full(sh, synth.as_u16(t["Q"]), synth.as_u16(t["K"]), synth.as_u16(t["V"]), d)["o"]
    rounded = torch.from_numpy(want).to(torch.bfloat16).double().numpy()
    assert np.linalg.norm(to_f64(O) - want) <= 1.02 * np.linalg.norm(rounded - want)


@pytest.mark.parametrize("D,n", [(128, 2), (128, 47), (128, 48), (128, 49), (64, 95), (64, 96), (64, 97), (128, 128),
                                 (128, 129), (64, 257)])
def test_combination_of_n_chunks(D, n):
    """Chunks of 256 keys around what a thread of the combination asks for ahead of the weights (48 or 96 chunks) and around
    its 128 threads.  The bound is the one above: rounding the result, and 2 % for the fp32 sums."""
    W, Lk = 255, 256 * n            # one chunk in the window, n - 1 before it
    t = synth.qkv(1, 1, 3, 1, D, seed=n, Lk=Lk)
    p = l2a.params(1, 1, Lk, 3, 1, D, W)
    ws = torch.full((l2a.l2a_decode_workspace_bytes(p),), 0x5A, dtype=torch.uint8, device="cuda")
    q, K, V = (t[k].cuda() for k in ("Q", "K", "V"))
    sh = oracle.Shape(1, 1, Lk, 3, 1, D, W)
    for routed in (1, 0):
        d = np.full((1, 1), routed, np.uint8)
        O = torch.full((1, 1, 3, D), float("nan"), dtype=torch.bfloat16, device="cuda")
        l2a.l2a_decode(p, q, K, V, torch.from_numpy(d[:, 0].copy()).cuda(), O, ws)
        assert l2a.l2a_workspace_status(ws) == 0
        want = oracle.forward_full(sh, synth.as_u16(t["Q"]), synth.as_u16(t["K"]), synth.as_u16(t["V"]), d)["o"]
        rounded = torch.from_numpy(want).to(torch.bfloat16).double().numpy()
        assert np.linalg.norm(to_f64(O) - want) <= 1.02 * np.linalg.norm(rounded - want), routed


def test_infinite_values_stay_infinite():
    """An infinite entry of V among the visible keys makes its column of the output infinite, and no other."""
    B, Lk, Hq, Hkv, D, W = 1, 700, 8, 2, 64, 200
    t = synth.qkv(B, 1, Hq, Hkv, D, seed=5, Lk=Lk)
    p = l2a.params(B, 1, Lk, Hq, Hkv, D, W)
    ws = torch.empty(l2a.l2a_decode_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    V = t["V"].clone()
    V[0, 690, 0, 3] = float("inf")
    V[0, 120, 1, 5] = -float("inf")          # before the window
    for d in (0, 1):
        O = torch.empty((B, 1, Hq, D), dtype=torch.bfloat16, device="cuda")
        l2a.l2a_decode(p, t["Q"].cuda(), t["K"].cuda(), V.cuda(), torch.tensor([d], dtype=torch.uint8, device="cuda"), O, ws)
        O = O.float().cpu()[0, 0]
        assert (O[:4, 3] == float("inf")).all()
        want = torch.isinf(O)
        want[:4, 3] = False
        assert want.sum() == (4 if d else 0) and (not d or (O[4:, 5] == -float("inf")).all()) and not torch.isnan(O).any()
