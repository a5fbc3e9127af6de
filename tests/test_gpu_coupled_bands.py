"""The coupled step's band heights (4 rows on small meshes, 7 on large ones) at
ragged row counts, against the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle as O
import pf_inputs as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,h,steps", [((3, 61), 1.0, 70), ((5, 59), (0.9, 1.1), 70),
                                           ((29, 121), 1.0, 130), ((1500, 1803), 1.0, 3),
                                           ((1499, 1805), (1.1, 0.9), 3)])
def test_coupled_bands(shape, h, steps):
    import paper_2601_06079_gb300 as pf
    U0 = G.coupled_initial(3, shape)
    s = pf.Solver(shape, h=h, model="coupled")
    s.set_params(kappa=0.3, mobility=1.0, mobility2=150.0, dt=1e-3)
    t = torch.from_numpy(U0).cuda()
    s.step_explicit(t, steps)
    P = O.Problem(shape, h=h, energy="coupled", kappa=0.3, mob=1.0, mob2=150.0)
    ref = P.coupled_explicit(U0, 1e-3, steps)
    got = t.cpu().numpy().astype(np.float64)
    for f in range(2):
        assert np.linalg.norm(got[f] - ref[f]) <= 1e-5 * np.linalg.norm(ref[f])
