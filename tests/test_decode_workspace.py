"""Decode workspace: sized once for a full cache and batch, it serves every earlier position and smaller batch; and the chunk
plan never asks for more than the size returned for its own shape."""
import random

import pytest

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

    def chunk(keys):
        per = -(-keys * B * Hkv // 296)
        return min(4096, max(256, -(-per // 64) * 64))

    return min(-(-win // chunk(win)), 64), min(-(-out // chunk(pos + 1)), 512)


def test_no_plan_exceeds_the_size():
    rng = random.Random(7)
    for _ in range(20000):
        Hkv, G, D = rng.choice([1, 2, 4, 8, 16]), rng.randint(1, 8), rng.choice([64, 128])
        B, W = rng.choice([1, 1, 2, 3, 7, 16, 40, 300]), rng.choice([0, 128, 1000, 4096, 100000])
        pos = int(2 ** rng.uniform(0, 20)) - 1
        rows = B * Hkv * sum(plan(B, pos, Hkv, W))
        done = -(-B * Hkv * 4 // 256) * 256
        need = 256 + done + -(-rows * G * (D + 4) * 4 // 256) * 256
        assert need <= size(B, pos + 1, pos, Hkv * G, Hkv, D, W), (B, pos, Hkv, G, D, W)
