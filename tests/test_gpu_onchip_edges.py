"""Explicit trajectories held on chip against one launch per step, bitwise, at the
edges that their tiles have: strips of 56 columns (32 pairs of columns less a halo
of 4 on each side), rows split over 16 warps, and the largest tiling (2048^2).
The fewest steps that go on chip are 8 + nodes / 2^18; what a call enqueues shows
that they did (the exchange buffer's zeroing and one kernel)."""
import ctypes as C

import pytest
import torch

import pf_inputs as G

pytestmark = pytest.mark.gpu

# widths around 1, 2 and 5 strips; heights around the rows of 16 warps and of
# several tiles; a mesh of 148 tiles of 512 rows
SHAPES = [(40, 55), (41, 56), (15, 57), (16, 111), (17, 112), (33, 113), (600, 279), (601, 280),
          (300, 281), (515, 1031), (2048, 2048)]


def solver(model, shape, form, stream=None):
    import paper_2601_06079_gb300 as pf
    s = pf.Solver(shape, model=model, stream=stream)
    s.set_params(W=1.0, kappa=0.5, mobility=1.0, dt=1e-3 if model == "ch" else 0.01)
    s.set_form(form)
    return s


def enqueued(s, stream, u, steps):
    """Operations of a call, counted as the nodes of its stream capture."""
    cuda = C.CDLL("libcuda.so.1")
    h, graph, n = C.c_void_p(stream.cuda_stream), C.c_void_p(), C.c_size_t()
    torch.cuda.synchronize()
    assert cuda.cuStreamBeginCapture_v2(h, 1) == 0  # thread-local
    s.step_explicit(u, steps)
    assert cuda.cuStreamEndCapture(h, C.byref(graph)) == 0
    assert cuda.cuGraphGetNodes(graph, None, C.byref(n)) == 0
    cuda.cuGraphDestroy(graph)
    return n.value


@pytest.mark.parametrize("model", ["ac", "ch"])
@pytest.mark.parametrize("shape", SHAPES)
def test_tile_edges(model, shape):
    least = 8 + (shape[0] * shape[1] >> 18)
    u0 = torch.from_numpy(G.ch_initial(11, shape)).cuda()
    stream = torch.cuda.Stream()
    chip = solver(model, shape, "fused_graph", stream)
    steps_form = solver(model, shape, "fused_stream")
    assert enqueued(chip, stream, u0.clone(), least) <= 2
    assert enqueued(chip, stream, u0.clone(), least - 1) > 2
    for steps in (least, least + 13):
        a, b = u0.clone(), u0.clone()
        torch.cuda.synchronize()
        chip.step_explicit(a, steps)
        stream.synchronize()
        steps_form.step_explicit(b, steps)
        assert torch.equal(a, b)


@pytest.mark.parametrize("model", ["ac", "ch"])
@pytest.mark.parametrize("shape,on_chip", [((600, 4300), False), ((1000, 3000), False),
                                           ((300, 8000), True), ((3000, 1000), True)])
def test_wide_meshes(model, shape, on_chip):
    # tiles of 56 columns and few of them down the mesh: 77 and 108 tall tiles take
    # longer than the band sweep, 143 and 144 low ones do not
    u0 = torch.from_numpy(G.ch_initial(12, shape)).cuda()
    stream = torch.cuda.Stream()
    s = solver(model, shape, "fused_graph", stream)
    assert (enqueued(s, stream, u0.clone(), 100) <= 2) == on_chip
    a, b = u0.clone(), u0.clone()
    torch.cuda.synchronize()
    s.step_explicit(a, 100)
    stream.synchronize()
    solver(model, shape, "fused_stream").step_explicit(b, 100)
    assert torch.equal(a, b)
