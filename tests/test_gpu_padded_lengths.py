"""Sequences of different lengths in one batch, right-padded to a common length.  Causal attention never looks at a
later key, so the rows of a shorter sequence are what a call at its own length gives, and with dO = 0 and d = 0 on the
padding rows (finite padding values) nothing flows back from them into dK, dV.  Bit for bit where both calls share key
blocks among as many CTAs and split key ranges alike (which follows from their numbers of key blocks and of groups of
routed rows, so from the batch); up to rounding elsewhere."""
import numpy as np
import pytest
import torch

from paper_2603_17484_b200 import l2a, synth
from tests.gpu_util import check_same_or_rounding, check_same_split, Case, run_backward

pytestmark = pytest.mark.gpu


def test_right_padded_batch_matches_single_sequences():
    Hq, Hkv, D, W = 4, 2, 128, 200
    lens = (1100, 517)
    L = max(lens)
    singles = []
    for i, n in enumerate(lens):
        d = synth.mask_bernoulli(1, n, 0.3, seed=60 + i)
        c = Case(1, n, Hq, Hkv, D, W, d, seed=70 + i, backward=True)
        c.run_forward()
        run_backward(c)
        singles.append(c)
    d = np.zeros((len(lens), L), np.uint8)
    for i, c in enumerate(singles):
        d[i, :lens[i]] = c.d[0]
    batch = Case(len(lens), L, Hq, Hkv, D, W, d, seed=99, backward=True)
    for name in ("Q", "K", "V", "dO"):
        t = getattr(batch.buf, name)
        t.zero_()                                  # finite padding; dO = 0 there
        for i, c in enumerate(singles):
            t[i, :lens[i]].copy_(getattr(c.buf, name)[0])
    batch.run_forward()
    run_backward(batch)
    for i, c in enumerate(singles):
        n = lens[i]
        for name in ("O", "dQ", "dK", "dV"):
            # bit-identical: same tiles and order of operations per row (at these sizes both calls take four CTAs per key
            # block and split no key range); a key block may see more query tiles than in the single call, but those are
            # masked or carry dO = 0 and add exact zeros
            got, want = getattr(batch.buf, name)[i, :n], getattr(c.buf, name)[0]
            if name == "dQ":   # summed over the key blocks with fp32 atomics: order not fixed
                check_same_or_rounding(got.contiguous(), want, name)
            else:
                assert torch.equal(got.contiguous().view(torch.int16), want.view(torch.int16)), (name, i)
        assert torch.all(batch.buf.dQ[i, n:] == 0) and torch.all(batch.buf.dK[i, n:] == 0)
        assert torch.all(batch.buf.dV[i, n:] == 0)


@pytest.mark.parametrize("lens,Hq,Hkv,D,split", [
    ((1100, 517, 1024), 8, 4, 128, "backward"),          # key blocks 36 (20, 32) alone: four CTAs each; 108 in the batch: two
    ((4500,) + (300,) * 8, 4, 1, 64, "forward"),         # 15 groups of routed rows alone, 36 key blocks: nine parts; 135: none
])
def test_padded_batch_across_the_lines_of_the_plan(lens, Hq, Hkv, D, split):
    """A batch in which another number of CTAs shares a key block, or key ranges are not split, than in the single calls."""
    W, L = 200, max(lens)
    d = np.zeros((len(lens), L), np.uint8)
    for i, n in enumerate(lens):
        d[i, :n] = synth.mask_bernoulli(1, n, 0.2, seed=160 + i)[0]
    backward = split == "backward"
    batch = Case(len(lens), L, Hq, Hkv, D, W, d, seed=199, backward=backward)
    batch.run_forward()
    if backward:
        for i, n in enumerate(lens):
            batch.buf.dO[i, n:].zero_()
        run_backward(batch)
    for i, n in enumerate(lens[:2]):
        c = Case(1, n, Hq, Hkv, D, W, d[i:i + 1, :n], seed=170 + i, backward=backward)
        names = ("Q", "K", "V") + (("dO",) if backward else ())
        for name in names:
            getattr(c.buf, name)[0].copy_(getattr(batch.buf, name)[i, :n])
        c.run_forward()
        rows = torch.from_numpy(d[i, :n].astype(bool)).cuda()
        got, want = batch.buf.O[i, :n], c.buf.O[0]
        assert torch.equal(got[~rows].view(torch.int16), want[~rows].view(torch.int16))     # rows that are not routed
        check_same_split(got[rows], want[rows], c.buf.V[0], "O")
        if backward:
            run_backward(c)
            for name in ("dQ", "dK", "dV"):
                check_same_or_rounding(getattr(batch.buf, name)[i, :n].contiguous(), getattr(c.buf, name)[0], name)
