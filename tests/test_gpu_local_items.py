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


def documents(L, lo, hi, seed):
    """int32 [n + 1] boundaries of documents of lo to hi tokens that fill L."""
    g = torch.Generator()
    g.manual_seed(seed)
    n = torch.randint(lo, hi + 1, (L // lo + 1,), generator=g)
    cu = torch.cat([torch.zeros(1, dtype=torch.int64), torch.cumsum(n, 0)])
    return torch.cat([cu[cu < L], torch.tensor([L])]).to(torch.int32)


@pytest.mark.parametrize("L,Lk,W,save,docs", [
    (32768, 32768, 0, True, None),            # items of one or two key blocks whose results, twice 268 MB, outlast them
    (32768, 32768, 128, True, None),
    (32768, 32768, 128, False, None),
    (16384, 16384, 4096, True, (16, 200)),    # short documents: ranges of keys from the table
    (16384, 16384, 4096, False, (16, 300)),
    (16384, 16384, 100, True, (200, 3000)),
    (3000, 5000, 64, True, None),             # queries behind cached keys; last group of a head with one tile
])
def test_short_items_hand_the_output_buffer_over(L, Lk, W, save, docs):
    """Items that end sooner than the store of the results before them.  Every output is that of calls over so few heads that
    each item has a CTA, bit for bit, time after time."""
    Hq, Hkv, D = 32, 8, 128
    g = torch.Generator(device="cuda")
    g.manual_seed(L + W)
    new = lambda *s: torch.empty(s, dtype=torch.bfloat16, device="cuda")
    Q, K, V = (new(1, n, h, D).normal_(generator=g) for n, h in ((L, Hq), (Lk, Hkv), (Lk, Hkv)))
    table = None if docs is None else l2a.l2a_pack_sequences(documents(L, *docs, seed=L + W).cuda(), L)
    flags = l2a.FLAG_SKIP_GLOBAL | (l2a.FLAG_SAVE_FOR_BWD if save else 0)

    def call(Q, K, V, O, S, lse, hq, hkv):
        st = ((L * Hq * D, Hq * D), (Lk * Hkv * D, Hkv * D)) if hq < Hq else (None, None)
        p = l2a.params(1, L, Lk, hq, hkv, D, W, flags=flags, q_stride=st[0], k_stride=st[1], v_stride=st[1], o_stride=st[0],
                       seq_bounds=table)
        ws = torch.empty(l2a.l2a_workspace_bytes(p)[1], dtype=torch.uint8, device="cuda")
        l2a.l2a_forward(p, Q, K, V, None, None, None, None, O, S, S, lse, lse, ws)
        return ws

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    groups = -(-L // 256)
    assert groups * Hq > sms
    want, want_lse = torch.full_like(Q, float("nan")), torch.empty((1, Hq, L), dtype=torch.float32, device="cuda")
    step = next(h for h in (4, 2, 1) if groups * h <= sms)
    for h0 in range(0, Hq, step):
        h, k = slice(h0, h0 + step), slice(h0 * Hkv // Hq, h0 * Hkv // Hq + 1)
        lse = torch.empty((1, step, L), dtype=torch.float32, device="cuda")
        ws = call(Q[:, :, h], K[:, :, k], V[:, :, k], want[:, :, h], new(1, L, step, D) if save else None, lse, step, 1)
        assert l2a.l2a_workspace_status(ws) == 0
        want_lse[:, h] = lse
    bits = want.view(torch.int16)
    assert torch.isfinite(want.float()).all()
    for _ in range(20):
        O, S = torch.full_like(Q, float("nan")), torch.full_like(Q, float("nan")) if save else None
        lse = torch.full_like(want_lse, float("nan"))
        ws = call(Q, K, V, O, S, lse, Hq, Hkv)
        assert l2a.l2a_workspace_status(ws) == 0
        assert torch.equal(O.view(torch.int16), bits)
        assert torch.equal(lse, want_lse)
        if save:
            assert torch.equal(S.view(torch.int16), bits)


def test_rows_whose_sequence_starts_behind_them():
    """A table that l2a_pack_sequences does not write: tiles of rows that see no key at all.  Their output is zero, the other
    rows are those of the call without such starts, and no wait runs out."""
    L, Hq, Hkv, D = 2048, 32, 8, 128
    Q, K, V = (torch.randn((1, L, h, D), device="cuda").to(torch.bfloat16) for h in (Hq, Hkv, Hkv))
    ws, out = None, []
    for shift in (0, 300):
        table = torch.tensor([[0, L]], dtype=torch.int32, device="cuda").repeat(L, 1)
        if shift:
            table[512:1024, 0] = torch.arange(512, 1024, dtype=torch.int32, device="cuda") + shift
        p = l2a.params(1, L, L, Hq, Hkv, D, 4096, flags=l2a.FLAG_SKIP_GLOBAL, seq_bounds=table)
        ws = torch.empty(l2a.l2a_workspace_bytes(p)[1], dtype=torch.uint8, device="cuda")
        O = torch.full_like(Q, float("nan"))
        l2a.l2a_forward(p, Q, K, V, None, None, None, None, O, None, None, None, None, ws)
        assert l2a.l2a_workspace_status(ws) == 0
        out.append(O)
    whole, holes = out
    assert not holes[:, 512:1024].any()
    for rows in (slice(0, 512), slice(1024, L)):
        assert torch.equal(holes[:, rows].view(torch.int16), whole[:, rows].view(torch.int16))
