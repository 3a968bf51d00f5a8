"""The two tiles of the local kernel that processes several items a CTA (attn_fwd_local.cu) stage their results in one buffer.
Every order in which the soft-max warps of both tiles and the store warp can go on is walked through here, with barriers that
are waited for by parity as mbarriers are: nothing may be overwritten before it has been stored, nobody may wait for good."""
import itertools
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_17484_b200", "csrc", "attn_fwd_local.cu")
TEXT = re.sub(r"//[^\n]*", "", open(SRC).read())


def walk(active1, wait_of, arrive_after, first):
    """active1: per item, whether its second tile has rows.  wait_of(t, k, use) -> (barrier, phase) that tile t waits for ahead
    of its k-th result, the use-th of both tiles, None: no wait; arrive_after(t, active1) -> barrier the store warp arrives at
    once a result has left; first: barrier it arrives at before anything.  Returns what went wrong, None: nothing."""
    uses = [(n, t) for n, a in enumerate(active1) for t in range(1 + a)]
    mine = [[u for u in uses if u[1] == t] for t in (0, 1)]
    number = {u: i for i, u in enumerate(uses)}
    barriers = sorted({"turn0", "turn1", "free"})
    zero = tuple(0 for _ in barriers)
    start = list(zero)
    if first is not None:
        start[barriers.index(first)] += 1
    # results staged by tile 0, by tile 1, stored ones, phases of the barriers, what the buffer holds (None: nothing to store)
    todo, seen = [(0, 0, 0, tuple(start), None)], set()
    while todo:
        s = todo.pop()
        if s in seen:
            continue
        seen.add(s)
        done0, done1, stored, phases, held = s
        moves = 0
        for t, k in ((0, done0), (1, done1)):
            if k == len(mine[t]):
                continue
            use = number[mine[t][k]]
            w = wait_of(t, k, use)
            if w is not None and (phases[barriers.index(w[0])] & 1) == (w[1] & 1):
                continue                                   # the phase of that parity is the one in progress: it waits
            moves += 1
            if held is not None:
                return "overwritten"
            todo.append((done0 + (t == 0), done1 + (t == 1), stored, phases, use))
        if stored < len(uses):
            n, t = uses[stored]
            if (done1 if t else done0) > mine[t].index((n, t)):       # staged
                moves += 1
                if held != stored:
                    return "overwritten"
                p = list(phases)
                p[barriers.index(arrive_after(t, active1[n]))] += 1
                todo.append((done0, done1, stored + 1, tuple(p), None))
        elif done0 == len(mine[0]) and done1 == len(mine[1]):
            continue
        if moves == 0:
            return "stuck"
    return None


PATTERNS = [p for n in range(1, 6) for p in itertools.product((0, 1), repeat=n)]


def test_turns():
    for p in PATTERNS:
        assert walk(p, lambda t, k, use: (f"turn{t}", k), lambda t, a: f"turn{1 if t < a else 0}", "turn0") is None, p


@pytest.mark.parametrize("name", ["every second phase", "nobody waits", "no first turn"])
def test_walk_finds_what_is_wrong(name):
    if name == "every second phase":       # one barrier, a phase per use, each tile waiting for the use before its own
        got = walk((1, 1, 1), lambda t, k, use: ("free", use - 1) if use else None, lambda t, a: "free", None)
        assert got == "overwritten"
    elif name == "nobody waits":
        assert walk((1, 1), lambda t, k, use: None, lambda t, a: "free", None) == "overwritten"
    else:
        assert walk((1, 1), lambda t, k, use: (f"turn{t}", k), lambda t, a: f"turn{1 if t < a else 0}", None) == "stuck"


def test_the_kernel_hands_the_buffer_over_in_turns():
    store = TEXT[TEXT.index("warp == kStoreWarp"):TEXT.index("warp > kMmaWarp")]
    softmax = TEXT[TEXT.index("warp > kMmaWarp"):TEXT.index("tmem_dealloc(tmem, 512);\n}")]
    assert re.search(r"mbar_init\(&bar->turn\[t\], 1\)", TEXT)
    assert re.findall(r"mbar_arrive\(&bar->turn\[([^;]*)\]\);", store) == ["0", "t < active1 ? 1 : 0"]
    assert store.index("mbar_arrive(&bar->turn[0])") < store.index("for (uint32_t n_items")
    assert store.index("tma_store_wait_read()") < store.index("turn[t < active1")
    # the wait for its turn: every result of the tile, its count as the phase, ahead of the stores into the buffer
    assert re.findall(r"mbar_wait\(&bar->turn([^,]*), ([^,]*), abort_flag\)", softmax) == [("[t]", "n_o & 1")]
    assert len(re.findall(r"\+\+n_o\b|\bn_o\+\+", softmax)) == 1
    order = [softmax.index(x) for x in ("bar->turn[t]", "st.shared.v4.b32", "fence_async_smem", "&bar->staged[t]", "++n_o")]
    assert order == sorted(order)
    assert "turn" not in TEXT[TEXT.index("warp == kTmaWarp"):TEXT.index("warp == kStoreWarp")].replace("return", "")
