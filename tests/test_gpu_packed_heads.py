"""Global pass and its backward over compact rows into which the query heads of a KV group are packed: numbers of rows (routed
tokens x heads of a group) at and around the edges of 128-row tiles and 256-row groups, against the fp64 oracle."""
import numpy as np
import pytest

from tests.gpu_util import Case, check_backward_full, run_backward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Hq,Hkv,D,n", [
    (7, 1, 128, 1), (7, 1, 128, 18), (7, 1, 128, 19), (7, 1, 128, 36), (7, 1, 128, 37),    # 7, 126, 133, 252, 259 rows
    (6, 2, 64, 43), (6, 2, 64, 85), (6, 2, 64, 86),                                        # 129, 255, 258
    (16, 2, 128, 16), (16, 2, 128, 32), (16, 2, 128, 33),                                  # 128, 256, 264
    (2, 2, 128, 128), (2, 2, 128, 129), (2, 2, 128, 300),                                  # one head a group; every token
])
@pytest.mark.parametrize("shared", [False, True])
def test_packed_heads(Hq, Hkv, D, n, shared):
    from paper_2603_17484_b200 import l2a
    L, B = 300, 2
    rng = np.random.default_rng(n)
    d = np.zeros((B, L), np.uint8)
    for b in range(B):                       # the second entry routes fewer tokens, the last one among them
        m = n if b == 0 else max(1, n // 3)
        d[b, rng.choice(L - 1, m - 1, replace=False)] = 1
        d[b, L - 1] = 1
    c = Case(B, L, Hq, Hkv, D, 40, d, seed=n, backward=True, flags=l2a.FLAG_SHARED_WINDOW if shared else 0)
    c.run_forward()
    c.check_forward_full()
    run_backward(c)
    check_backward_full(c)
