"""The index-checking build of the library: indices far outside of the queries are reported, their rows are neither read nor
stored, and all other rows are those of a run without them."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys
sys.path.insert(0, sys.argv[1])
import torch
from paper_2603_17484_b200 import build, l2a, synth
l2a.LIB_PATH = build.build_lib(debug=True)
assert "debug" in l2a.version()
from tests.gpu_util import Case

for D, Hq, Hkv in ((128, 4, 2), (64, 3, 1)):
    B, L, W = 1, 600, 64
    d = synth.mask_bernoulli(B, L, 0.3, seed=4)
    c = Case(B, L, Hq, Hkv, D, W, d, seed=8, backward=True)
    b = c.run_forward()
    n, want, idx = int(b.n_routed[0]), b.O.clone(), b.q_idx.clone()
    bad = {n // 2: -1, n - 1: 2 * L + 5}
    for k, v in bad.items():
        b.q_idx[0, k] = v
    b.O.fill_(float("nan"))
    b.forward()
    torch.cuda.synchronize()
    assert l2a.l2a_workspace_status(b.fwd_ws) == -6
    assert b.check_guards()
    rest = torch.ones(L, dtype=torch.bool, device="cuda")
    for k in bad:
        rest[idx[0, k].long()] = False
    assert torch.equal(b.O[0, rest], want[0, rest])
    assert torch.equal(b.O[0, ~rest], b.S_save[0, ~rest])
print("GATHER_CHECKS_OK")
"""


def test_gather_checks_its_indices():
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "GATHER_CHECKS_OK" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
