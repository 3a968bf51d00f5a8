"""A quarter of the forward's probabilities comes from a polynomial on the FMA pipe instead of ex2: its error bound and its
edge values, on the CPU with the constants of the source, and on the GPU through the log-sum-exp of rows whose visible keys
all take it."""
import os
import re

import numpy as np
import pytest
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
BOUND = 2.2e-7           # as the source states it
F = np.float32


def _source():
    text = open(os.path.join(ROOT, "paper_2603_17484_b200", "csrc", "sm100_prims.cuh")).read()
    body = text[text.index("float2 exp2_fma2(float2 x)"):]
    return body[:body.index("\n}")]


def _coefficients():
    """c5 .. c0 in the order of the Horner steps."""
    c = [F(v) for v in re.findall(r"make_float2\((0\.\d+|1\.\d+)f, \1f\)", _source())]
    assert len(c) == 6
    return c


def _fma(a, b, c):
    """float32 fused multiply-add: the product of two float32 is exact in float64, so only the last step can round twice."""
    return (a.astype(np.float64) * np.float64(b) + np.asarray(c, np.float64)).astype(F)


def exp2_fma(x):
    shift = F(12583039.0)                                   # 1.5 * 2^23 + 127
    assert "12583039.f" in _source() and "-127.f" in _source()
    with np.errstate(invalid="ignore", over="ignore"):
        x = np.where(np.isnan(x), x, np.maximum(x, F(-127)))
        t = (x + shift).astype(F)
        n = (t - shift).astype(F)
        f = _fma(n, F(-1), x)
        c = _coefficients()
        p = np.full_like(f, c[0])
        for k in c[1:]:
            p = (p.astype(np.float64) * f.astype(np.float64) + np.float64(k)).astype(F)
        scale = (t.view(np.uint32) << np.uint32(23)).view(F)
        return (p * scale).astype(F)


def test_coefficients_are_the_minimax_fit():
    """Remez exchange for the relative error of 2^f on [-1/2, 1/2]."""
    g = np.linspace(-0.5, 0.5, 100001)
    x = 0.5 * np.cos(np.pi * np.arange(7) / 6)[::-1]
    for _ in range(8):
        rows = np.concatenate([x[:, None] ** np.arange(6) / 2.0 ** x[:, None], (-1.0) ** np.arange(7)[:, None]], axis=1)
        c = np.linalg.solve(rows, np.ones(7))[:6]
        e = np.polynomial.polynomial.polyval(g, c) / 2.0 ** g - 1
        change = np.flatnonzero(np.diff(np.sign(e))) + 1
        x = np.array([p[np.abs(q).argmax()] for p, q in zip(np.split(g, change), np.split(e, change))])
    want = c[::-1].astype(F)
    got = np.array(_coefficients())
    assert (np.abs(got - want) <= np.spacing(want)).all()


def test_error_bound():
    x = np.concatenate([np.linspace(-126, 8, 3_000_001), -np.logspace(-8, 2, 400_001), np.logspace(-8, 0.9, 100_001),
                        np.arange(-126, 9), np.arange(-125.5, 8)]).astype(F)
    want = np.exp2(x.astype(np.float64))
    rel = np.abs(exp2_fma(x).astype(np.float64) - want) / want
    assert rel.max() <= BOUND, (rel.max(), x[rel.argmax()])


def test_edges():
    x = np.array([-np.inf, -1e30, -127.0, -126.75, np.nan, 0.0], F)
    got = exp2_fma(x)
    assert list(got[:4]) == [0.0] * 4 and np.isnan(got[4]) and abs(got[5] - 1) <= BOUND
    # results of the half octave below 2^-126 are subnormal, with their spacing of 2^-149
    x = np.linspace(-126.499, -126, 10001).astype(F)
    got = exp2_fma(x).astype(np.float64)
    assert (np.abs(got - np.exp2(x.astype(np.float64))) <= 2.0 ** -149 + BOUND * 2.0 ** -126).all()


@pytest.mark.gpu
def test_polynomial_on_the_gpu():
    """Of every eight keys the last two take the polynomial.  Their scores lie in [-5, 0]; key 0 has score 0, the others
    exponentials of exactly zero.  The fp32 log-sum-exp of a row then is log(1 + the sum of its polynomial values)."""
    from paper_2603_17484_b200 import l2a

    L, D = 128, 64
    p = l2a.params(1, L, L, 1, 1, D, L, softmax_scale=1.0, flags=0)
    b = l2a.Buffers.allocate(p)
    b.lse_loc = torch.empty(1, 1, L, dtype=torch.float32, device="cuda")
    # scores q . k in the natural-log domain: q = (1, 1, 0, ...), k = (hi, lo, 0, ...) with both parts exact in bf16
    s = -torch.linspace(0.01, 5.0, L, dtype=torch.float64)
    hi = s.to(torch.bfloat16)
    lo = (s - hi.double()).to(torch.bfloat16)
    col = torch.arange(L) % 8
    hi[(col < 6)] = -16384.0
    lo[(col < 6)] = 0.0
    hi[0] = lo[0] = 0.0
    for t in (b.Q, b.K, b.V):
        t.zero_()
    b.Q[0, :, 0, :2] = 1.0
    b.K[0, :, 0, 0] = hi.cuda()
    b.K[0, :, 0, 1] = lo.cuda()
    b.router.zero_()
    b.route()
    b.forward()
    torch.cuda.synchronize()
    score = hi.double() + lo.double()
    e = torch.exp(score)
    want = torch.log(torch.cumsum(e, 0))
    got = b.lse_loc[0, 0].double().cpu()
    # relative error of a polynomial value: 2.2e-7, and ln 2 times that of its argument (log2(e) in fp32: 5 x 2e-8, one
    # rounding below 8: 2^-22); of the sum of up to 33 terms: 2^-24 an addition; logarithm and its scaling: 3 x 2^-24 of 4
    bound = 2.2e-7 + 0.7 * (1e-7 + 2.0 ** -22) + 33 * 2.0 ** -24 + 12 * 2.0 ** -24
    assert float((got - want).abs().max()) <= bound, float((got - want).abs().max())
