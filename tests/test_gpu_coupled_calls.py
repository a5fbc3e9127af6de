"""What a call of the coupled step enqueues, besides its steps."""
import ctypes as C

import pytest
import torch

import pf_inputs as G

pytestmark = pytest.mark.gpu


def solver(stream=None, shape=(48, 70)):
    import paper_2601_06079_gb300 as pf
    s = pf.Solver(shape, model="coupled", stream=stream)
    s.set_params(kappa=0.3, mobility=1.0, mobility2=150.0, dt=1e-3)
    return s


def test_short_run_takes_two_launches_beside_its_steps():
    # launches of a short run, counted as the nodes of its stream capture
    cuda = C.CDLL("libcuda.so.1")
    stream = torch.cuda.Stream()
    s = solver(stream)
    u = torch.from_numpy(G.coupled_initial(3, (48, 70))).cuda()
    s.step_explicit(u, 20)
    torch.cuda.synchronize()
    h, graph, n = C.c_void_p(stream.cuda_stream), C.c_void_p(), C.c_size_t()
    assert cuda.cuStreamBeginCapture_v2(h, 1) == 0  # thread-local
    s.step_explicit(u, 20)
    assert cuda.cuStreamEndCapture(h, C.byref(graph)) == 0
    assert cuda.cuGraphGetNodes(graph, None, C.byref(n)) == 0
    cuda.cuGraphDestroy(graph)
    assert n.value == 22


@pytest.mark.parametrize("shape,steps", [((48, 70), 20), ((48, 70), 64), ((48, 70), 150),
                                         ((1400, 1501), 40)])
def test_call_can_be_captured(shape, steps):
    # also: steps that overlap the launch before them against steps that do not
    stream = torch.cuda.Stream()
    s = solver(stream, shape)
    u0 = torch.from_numpy(G.coupled_initial(3, shape)).cuda()
    a, b = u0.clone(), u0.clone()
    torch.cuda.synchronize()
    s.step_explicit(a, steps)
    stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        s.step_explicit(b, steps)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(a, b)
