"""dLoss/dM near its zero.  dLoss/dM = (kappa dLoss/dkappa + W dLoss/dW) / M, and
the two parts, of opposite sign, nearly cancel at these step counts (by a factor
of 12 to 1,600), so that a relative difference between them shows.

Bars.  One coefficient of the step off by 3e-8 (half a unit of FP32 at the upper
end of a binade) shifts dLoss/dM by 1e-8 or more of |kappa dLoss/dkappa| +
|W dLoss/dW|, evaluated in FP64; the rounding of the states is random over nodes
and steps and far below.  On square cells no factor is left rounded: 1e-8.  On
others the stencil's side weights are: 3e-8.  The two parts themselves: 1e-7."""
import numpy as np
import pytest
import torch

import oracle as O
import pf_inputs as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,h,steps,bar", [((66, 78), 1.0, 250, 1e-8),
                                               ((66, 78), 1.0, 270, 1e-8),
                                               ((120, 125), 1.0, 330, 1e-8),
                                               ((41, 70), (1.25, 0.8), 200, 3e-8),
                                               ((41, 70), (1.25, 0.8), 250, 3e-8)])
def test_mobility_gradient_near_its_zero(shape, h, steps, bar):
    import paper_2601_06079_gb300 as pf
    mob = G.gaussian_mobility(3, shape, h=1.0, width=(16.0, 32.0)).astype(np.float32)
    c0 = G.ch_initial(4, shape)
    y, x = np.mgrid[:shape[0], :shape[1]]
    target = (0.5 + 0.03 * np.sin(0.3 * x + 1) * np.sin(0.25 * y + 2)).astype(np.float32)
    s = pf.Solver(shape, h=h, model="ch")
    s.set_params(W=1.0, kappa=0.5, mobility=1.0, dt=1e-3, mobility_field=torch.from_numpy(mob))
    _, g = s.adjoint(torch.from_numpy(c0).cuda(), torch.from_numpy(target).cuda(), steps, 50)
    P = O.Problem(shape, h=h, W=1.0, kappa=0.5, mob=1.0, mob_field=mob.astype(np.float64))
    _, ref = P.ch_adjoint(c0, target, 1e-3, steps)
    parts = abs(0.5 * ref["kappa"]) + abs(ref["W"])
    for k in ("kappa", "W"):
        assert abs(g[k] - ref[k]) <= 1e-7 * abs(ref[k]), k
    assert abs(g["M"] - ref["M"]) <= bar * parts
