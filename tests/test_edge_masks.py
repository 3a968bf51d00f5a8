"""Edge tiles: the keys a row sees, and the rows that see a key, are taken as one range each (bits of a tile's 32 columns).
CPU restatement of the two rules against the definition of the mask, for every mode that reaches the kernels; GPU runs
with windows and offsets around the 32-column and 128-row tile edges against the fp64 oracle."""
import numpy as np
import pytest

from paper_2603_17484_b200 import synth


def _mask(n, lk, w, off, shift, start):
    """[row, key]: key visible to row; shift > 0: only keys before the window (shared-window global pass)."""
    pos = np.arange(n)[:, None] + off
    k = np.arange(lk)[None, :]
    return (k <= pos - shift) & (k >= (pos - w if w is not None else -1)) & (k >= start[:, None])


@pytest.mark.parametrize("seed", range(20))
def test_ranges_equal_the_mask(seed):
    rng = np.random.default_rng(seed)
    packed = seed % 2 == 1
    n = int(rng.integers(1, 400))
    off = 0 if packed else int(rng.integers(0, 150))
    lk = n + off if packed else n + off + int(rng.integers(0, 3))
    w = int(rng.choice([0, 1, 31, 32, 127, 128, 129, 500]))
    start, end = np.zeros(n, int), np.full(n, n)
    if packed:
        cuts = np.unique(np.concatenate([[0, n], rng.integers(0, n + 1, 5)]))
        for s, e in zip(cuts[:-1], cuts[1:]):
            start[s:e], end[s:e] = s, e
    q_idx = np.flatnonzero(rng.random(n) < 0.3)
    prefix = np.concatenate([[0], np.cumsum(np.isin(np.arange(n), q_idx))])
    for shift in (0, w + 1):
        loc = _mask(n, lk, w, off, 0, start)
        glb = _mask(n, lk, None, off, shift, start)[q_idx]
        for kp in range(lk + 5):                                   # keys past the end: the ragged last block
            row_end = (int(end[kp]) if kp < n else 0) if packed else n
            first = min(max(kp - off, 0), n)
            last = min(kp + w - off + 1, row_end)
            want = loc[:, kp] if kp < lk else np.zeros(n, bool)
            assert np.array_equal(want, (np.arange(n) >= first) & (np.arange(n) < last)), (kp, "local")
            c0 = prefix[min(max(kp - off + shift, 0), n)]
            c1 = prefix[row_end] if row_end < n else len(q_idx)
            want = glb[:, kp] if kp < lk else np.zeros(len(q_idx), bool)
            c = np.arange(len(q_idx))
            assert np.array_equal(want, (c >= c0) & (c < c1)), (kp, "global")
        for r in range(n):                                         # forward: a row's keys
            k = np.arange(lk)
            assert np.array_equal(loc[r], (k >= max(r + off - w, start[r])) & (k < r + off + 1))


@pytest.mark.gpu
@pytest.mark.parametrize("W", [0, 31, 32, 127, 128, 129])
@pytest.mark.parametrize("L,Lk,D", [(257, 257, 128), (300, 427, 64)])
def test_edges_on_the_gpu(W, L, Lk, D):
    from tests.gpu_util import Case, check_backward_full, run_backward
    d = synth.mask_bernoulli(1, L, 0.4, seed=W)
    c = Case(1, L, 2, 1, D, W, d, seed=W + 1, Lk=Lk, backward=True)
    c.run_forward()
    c.check_forward_full()
    run_backward(c)
    check_backward_full(c)
