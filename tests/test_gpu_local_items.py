"""The local pass of more work items (256 rows of a head) than SMs runs on CTAs that take one item after the other, fewer items
get a CTA each.  Both do the same arithmetic: a call over all heads gives the bits of calls over a few heads each."""
import pytest
import torch

from paper_2603_17484_b200 import l2a

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,L,Hq,Hkv,W,save", [
    (1, 128, 152, 8, 40, False),       # few items more than SMs, second tile without rows
    (1, 129, 300, 4, 4096, True),      # second tile with one row; more than two items a CTA
    (1, 257, 160, 8, 100, True),       # last item of a head: one row
    (3, 700, 64, 8, 4096, False),      # ragged rows, several sequences
    (2, 1024, 64, 16, 0, True),        # a window of one key
    (1, 5000, 40, 8, 1000, True),      # band edges, several key blocks an item, 800 items
])
def test_many_items_equal_few(B, L, Hq, Hkv, W, save):
    D = 128
    g = torch.Generator(device="cuda")
    g.manual_seed(L + Hq)
    new = lambda *s: torch.empty(s, dtype=torch.bfloat16, device="cuda")
    Q, K, V = new(B, L, Hq, D).normal_(generator=g), new(B, L, Hkv, D).normal_(generator=g), new(B, L, Hkv, D).normal_(generator=g)
    flags = l2a.FLAG_SKIP_GLOBAL | (l2a.FLAG_SAVE_FOR_BWD if save else 0)

    def call(Q, K, V, O, hq, hkv):
        strided = ((L * Hq * D, Hq * D), (L * Hkv * D, Hkv * D)) if hq < Hq else (None, None)
        p = l2a.params(B, L, L, hq, hkv, D, W, flags=flags, q_stride=strided[0], k_stride=strided[1], v_stride=strided[1],
                       o_stride=strided[0])
        S = new(B, L, hq, D) if save else None
        lse = torch.full((B, hq, L), float("nan"), dtype=torch.float32, device="cuda")
        A = new(B, L, hq, D) if save else None
        ws = torch.empty(l2a.l2a_workspace_bytes(p)[1], dtype=torch.uint8, device="cuda")
        l2a.l2a_forward(p, Q, K, V, None, None, None, None, O, S, A, lse, torch.empty_like(lse) if save else None, ws)
        assert l2a.l2a_workspace_status(ws) == 0
        return S, lse

    whole, parts = torch.full_like(Q, float("nan")), torch.full_like(Q, float("nan"))
    S, lse = call(Q, K, V, whole, Hq, Hkv)
    assert -(-L // 256) * Hq * B > torch.cuda.get_device_properties(0).multi_processor_count
    if save:
        assert torch.equal(S.view(torch.int16), whole.view(torch.int16))
    G = Hq // Hkv
    for g0 in range(Hkv):
        for h0 in range(0, G, 5):          # at most five heads: -(-5000 // 256) * 5 = 100 items
            h = slice(g0 * G + h0, min(g0 * G + h0 + 5, (g0 + 1) * G))
            k = slice(g0, g0 + 1)
            _, lse_part = call(Q[:, :, h], K[:, :, k], V[:, :, k], parts[:, :, h], h.stop - h.start, 1)
            assert torch.equal(lse_part, lse[:, h])
    assert torch.equal(whole.view(torch.int16), parts.view(torch.int16))
