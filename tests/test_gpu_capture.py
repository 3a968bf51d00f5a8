"""The launches of a step overlap (programmatic dependent launches): captured into a CUDA graph, on a stream of their own,
and repeated without a synchronisation in between, they give the bits of single calls."""
import ctypes

import pytest
import torch

from paper_2603_17484_b200 import l2a, synth
from tests.gpu_util import Case, check_same_or_rounding, run_backward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,Hq,Hkv,flags", [(700, 4, 2, 0), (4500, 2, 1, 0), (700, 4, 2, l2a.FLAG_SHARED_WINDOW),
                                             (4500, 12, 2, 0)])     # 216 local items: more than SMs
def test_captured_step_equals_single_calls(L, Hq, Hkv, flags):
    D, W = 128, 200
    inputs = [Case(1, L, Hq, Hkv, D, W, synth.mask_bernoulli(1, L, rho, seed=3 + i), seed=20 + i, backward=True, flags=flags)
              for i, rho in enumerate((0.3, 0.1))]
    names = ("O", "dK", "dV", "dQ", "q_idx", "n_routed")
    want = []
    for c in inputs:
        c.run_forward()
        run_backward(c, with_dgate=False)
        want.append({n: getattr(c.buf, n).clone() for n in names})
    work = Case(1, L, Hq, Hkv, D, W, inputs[0].d, seed=20, backward=True, flags=flags)
    b = work.buf
    stream = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()

    def step():
        b.route(work.kind)
        b.forward()
        b.backward()

    def load(c):
        for n in ("Q", "K", "V", "dO", "router"):
            getattr(b, n).copy_(getattr(c.buf, n))

    with torch.cuda.stream(stream):
        step()
        with torch.cuda.graph(graph, stream=stream):
            step()
        for run in (graph.replay, step):
            for k in (0, 1, 0):
                load(inputs[k])
                for _ in range(3):            # back to back: a step must not start before the last one's readers are done
                    run()
                got = {n: getattr(b, n).clone() for n in names}
                for n in names:
                    if n == "dQ":             # fp32 atomics: order not fixed
                        check_same_or_rounding(got[n], want[k][n], n)
                    else:
                        assert torch.equal(got[n].view(torch.int32 if got[n].dtype == torch.int32 else torch.int16),
                                           want[k][n].view(torch.int32 if got[n].dtype == torch.int32 else torch.int16)), (n, k)
    torch.cuda.synchronize()
    assert l2a.l2a_workspace_status(b.fwd_ws) == 0 and l2a.l2a_workspace_status(b.bwd_ws) == 0
    assert b.check_guards()


def test_global_pass_overlaps_only_a_plainly_launched_local_pass():
    """The global pass reads the routing and the compacted queries before it waits for the local pass.  So the local pass,
    the only kernel it may overlap with, has to be behind the gather by a full dependency (captured, not run)."""
    cuda = ctypes.CDLL("libcuda.so.1")
    c = Case(1, 300, 2, 1, 128, 64, synth.mask_bernoulli(1, 300, 0.3, seed=1), seed=2)
    stream = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g, stream=stream):
        c.buf.forward()
    graph = ctypes.c_void_p(g.raw_cuda_graph())
    n = ctypes.c_size_t(0)
    assert cuda.cuGraphGetEdges_v2(graph, None, None, None, ctypes.byref(n)) == 0
    assert n.value == 2                                   # gather -> local -> global
    src, dst, data = (ctypes.c_void_p * 2)(), (ctypes.c_void_p * 2)(), (ctypes.c_uint8 * 16)()    # 8 bytes an edge
    assert cuda.cuGraphGetEdges_v2(graph, src, dst, data, ctypes.byref(n)) == 0
    first = 0 if dst[0] == src[1] else 1
    assert dst[first] == src[1 - first]
    assert data[8 * first] == 0                           # from_port: full completion of the gather
    assert data[8 * (1 - first)] == 1                     # programmatic: the global pass starts under the local one
