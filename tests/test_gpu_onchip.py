"""Trajectories held on chip (the default form of explicit 2-D runs that fit)
against one launch per step: bitwise equal, at tile edges and remainders."""
import pytest
import torch

import pf_inputs as G

pytestmark = pytest.mark.gpu

# one tile; ragged strips at one and two pairs per lane (60 / 120 columns for
# Cahn-Hilliard, 64 / 128 for Allen-Cahn); odd widths; fewer rows than warps;
# many tiles in both directions; the largest mesh of the range
SHAPES = [(3, 3), (4, 5), (64, 64), (17, 61), (33, 119), (40, 121), (7, 127), (16, 129),
          (129, 515), (515, 1031), (1500, 37), (37, 1501), (2048, 2048)]


def run(model, shape, form, steps, **kw):
    import paper_2601_06079_gb300 as pf
    h = kw.pop("h", 1.0)
    s = pf.Solver(shape, h=h, model=model)
    s.set_params(W=1.0, kappa=0.5, mobility=1.0, dt=1e-3 if model == "ch" else 0.01, **kw)
    s.set_form(form)
    u = torch.from_numpy(G.ch_initial(11, shape)).cuda()
    s.step_explicit(u, steps)
    return u


@pytest.mark.parametrize("model", ["ac", "ch"])
@pytest.mark.parametrize("shape", SHAPES)
def test_onchip_is_bitwise_the_stepwise_form(model, shape):
    for steps in (8, 21):
        a, b = (run(model, shape, f, steps) for f in ("fused_graph", "fused_stream"))
        assert torch.equal(a, b)


@pytest.mark.parametrize("model", ["ac", "ch"])
@pytest.mark.parametrize("kw", [dict(h=(0.8, 1.25)), dict(shift=0.45),
                                dict(h=(1.2, 0.9), shift=0.4)])
def test_onchip_general_coefficients(model, kw):
    a, b = (run(model, (70, 131), f, 40, **kw) for f in ("fused_graph", "fused_stream"))
    assert torch.equal(a, b)


def test_smallest_allen_cahn_meshes():
    for shape in ((2, 2), (2, 9), (9, 2), (2, 300), (300, 2)):
        a, b = (run("ac", shape, f, 33) for f in ("fused_graph", "fused_stream"))
        assert torch.equal(a, b)
