"""Decode workspace: sized once for a full cache and batch, it serves every earlier position and smaller batch; and the chunk
plan never asks for more than the size returned for its own shape."""
import ctypes
import random

import pytest
import torch

from paper_2603_17484_b200 import build as l2a_build
from paper_2603_17484_b200 import l2a


def size(B, Lk, pos, Hq, Hkv, D, W):
    return l2a.l2a_decode_workspace_bytes(l2a.params(B, 1, Lk, Hq, Hkv, D, W, q_pos_offset=pos))


@pytest.fixture(scope="module", autouse=True)
def _lib():
    l2a_build.build_lib()


@pytest.mark.parametrize("B,Hq,Hkv,D,W,cap", [
    (1, 28, 4, 128, 4096, 131072),     # 89 chunks at 3642 earlier positions, 88 at the last
    (1, 32, 8, 128, 1000, 10240),      # 38 and 33
    (16, 32, 8, 128, 4096, 131072),
    (7, 12, 2, 64, 100000, 140000),    # window larger than most of the cache
    (300, 8, 1, 64, 128, 5000),
])
def test_size_at_capacity_is_enough_for_earlier_positions(B, Hq, Hkv, D, W, cap):
    full = size(B, cap, cap - 1, Hq, Hkv, D, W)
    step = 1 if cap <= 20000 else 7
    for pos in list(range(0, cap, step)) + [cap - 2]:
        assert size(B, cap, pos, Hq, Hkv, D, W) <= full, pos                  # cache allocated ahead
    for pos in range(0, cap, 61):
        assert size(B, pos + 1, pos, Hq, Hkv, D, W) <= full, pos              # a view of the keys so far
    for b in range(1, B):
        assert size(b, cap, cap - 1, Hq, Hkv, D, W) <= full, b                # sequences that have ended left the batch


def plan(B, pos, Hkv, W):
    """Chunks per (sequence, KV head), restated: inside the window, before it."""
    win = min(pos, W) + 1
    out = pos + 1 - win

    def chunk(keys, target, least):
        return min(4096, max(least, -(-(-(-keys // target)) // 64) * 64))

    length = min(chunk((pos + 1) * Hkv, 148, 1536), chunk((pos + 1) * B * Hkv, 296, 256))
    return min(-(-win // chunk(win * B * Hkv, 296, 256)), 64), min(-(-out // length), 512)


def plan_bytes(B, pos, Hq, Hkv, D, W):
    rows = B * Hkv * sum(plan(B, pos, Hkv, W))
    return 256 + -(-B * Hkv * 4 // 256) * 256 + -(-rows * (Hq // Hkv) * (D + 4) * 4 // 256) * 256


@pytest.mark.skipif(torch.cuda.is_available(), reason="passes addresses that only a machine without a device may see")
@pytest.mark.parametrize("B,L,Hkv,W", [(16, 32768, 4, 4096), (32, 60000, 1, 4096), (16, 131072, 1, 4096), (32, 16384, 4, 4096),
                                       (16, 32768, 8, 4096), (1, 131072, 8, 4096), (8, 30000, 2, 128)])
def test_one_routed_sequence_gives_work_to_many_sms(B, L, Hkv, W):
    """Whatever the batch: chunks for half the SMs, or of no more than 1536 keys.  The library asks for the workspace of no
    less than this plan (it refuses one byte less before it touches anything)."""
    n_win, n_out = plan(B, L - 1, Hkv, W)
    assert Hkv * (n_win + n_out) >= 74 or -(-(L - W - 1) // n_out) <= 1536
    p = l2a.params(B, 1, L, Hkv, Hkv, 64, W)
    some = 1 << 20
    assert l2a.lib().l2a_decode(ctypes.byref(p), some, some, some, None, some, some,
                                plan_bytes(B, L - 1, Hkv, Hkv, 64, W) - 1, None) == -3


def test_no_plan_exceeds_the_size():
    rng = random.Random(7)
    for _ in range(20000):
        Hkv, G, D = rng.choice([1, 2, 4, 8, 16]), rng.randint(1, 8), rng.choice([64, 128])
        B, W = rng.choice([1, 1, 2, 3, 7, 16, 40, 300]), rng.choice([0, 128, 1000, 4096, 100000])
        pos = int(2 ** rng.uniform(0, 20)) - 1
        assert plan_bytes(B, pos, Hkv * G, Hkv, D, W) <= size(B, pos + 1, pos, Hkv * G, Hkv, D, W), (B, pos, Hkv, G, D, W)
